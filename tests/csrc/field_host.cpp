// Error of the FP64 field map (emt_field.cuh) and of the RK4 stages it stands
// for (the oracle's operation order), both in FP64, against the stages in
// 113-bit arithmetic: n equal substeps of turn t from the origin, tracks of
// random direction, charge and bending radius, every fourth within a few
// degrees of the field.  Position errors are in units of the bending radius.
// Prints per case: t, n, axis (-1: any direction), then the rms and the
// largest position and direction error of the map and of the stages.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>

#include "../../paper_2203_09467_gb300/csrc/emt_field.cuh"

#if defined(__SIZEOF_FLOAT128__)
typedef __float128 quad;
#else
typedef long double quad;  // 113 bits where __float128 is missing (AArch64)
#endif

static uint64_t g_s = 0x9E3779B97F4A7C15ull;
static double uniform()
{
    g_s ^= g_s << 13;
    g_s ^= g_s >> 7;
    g_s ^= g_s << 17;
    return (double)(g_s >> 11) * 0x1p-53;
}

static double madd(double a, double b, double c) { return fma(a, b, c); }
static quad madd(quad a, quad b, quad c) { return a * b + c; }
static double root(double a) { return sqrt(a); }
static quad root(quad a)
{
    quad r = sqrt((double)a);
    for (int k = 0; k < 3; ++k) r = (r + a / r) / 2;
    return r;
}

template <typename T>
static void slope(const T v[3], const T B[3], T kq, T a[3])
{
    for (int i = 0; i < 3; ++i) {
        const int j = (i + 1) % 3, k = (i + 2) % 3;
        a[i] = kq * madd(v[j], B[k], -(v[k] * B[j]));
    }
}

template <typename T>
static void stages(T kq, const T B[3], T h, T x[3], T u[3])
{
    T a1[3], a2[3], a3[3], a4[3], u2[3], u3[3], u4[3];
    const T hh = T(0.5) * h, h6 = h / T(6);
    slope(u, B, kq, a1);
    for (int i = 0; i < 3; ++i) u2[i] = madd(hh, a1[i], u[i]);
    slope(u2, B, kq, a2);
    for (int i = 0; i < 3; ++i) u3[i] = madd(hh, a2[i], u[i]);
    slope(u3, B, kq, a3);
    for (int i = 0; i < 3; ++i) u4[i] = madd(h, a3[i], u[i]);
    slope(u4, B, kq, a4);
    for (int i = 0; i < 3; ++i) {
        x[i] = madd(h6, madd(T(2), u3[i], madd(T(2), u2[i], u[i])) + u4[i], x[i]);
        u[i] = madd(h6, madd(T(2), a3[i], madd(T(2), a2[i], a1[i])) + a4[i], u[i]);
    }
    const T n = root(madd(u[0], u[0], madd(u[1], u[1], u[2] * u[2])));
    for (int i = 0; i < 3; ++i) u[i] = u[i] / n;
}

struct Field {
    int baxis;
    double B[3], bmag, bhat[3];
};

struct Error {
    double sum = 0.0, most = 0.0;
    void add(const double a[3], const quad b[3], double unit)
    {
        quad s = 0;
        for (int i = 0; i < 3; ++i) s += ((quad)a[i] - b[i]) * ((quad)a[i] - b[i]);
        const double d = sqrt((double)s) / unit;
        sum += d * d;
        if (!(d <= most)) most = d;
    }
};

int main(int argc, char** argv)
{
    const int tracks = argc > 1 ? atoi(argv[1]) : 150;
    const double turns[] = {0.002, 0.005, 0.02, 0.035, 0.05, 0.085, 0.12, 0.2, 0.3, 0.4, 0.5};
    const int counts[] = {1, 2, 7, 30, 100};
    for (double turn : turns)
        for (int n : counts)
            for (int axis = -1; axis < 3; ++axis) {
                Error e[4];  // position and direction: map, stages
                for (int k = 0; k < tracks; ++k) {
                    Field f{axis, {0, 0, 0}, 0, {0, 0, 0}};
                    if (axis >= 0)
                        f.B[axis] = 1.0 + 2.0 * uniform();
                    else
                        for (double& b : f.B) b = 4.0 * uniform() - 2.0;
                    f.bmag = sqrt(f.B[0] * f.B[0] + f.B[1] * f.B[1] + f.B[2] * f.B[2]);
                    for (int i = 0; i < 3; ++i) f.bhat[i] = f.B[i] / f.bmag;
                    const double radius = 0.5 * exp(5.0 * uniform());
                    const double kq = (uniform() < 0.5 ? -1.0 : 1.0) / (radius * f.bmag);
                    const double h = turn * radius * (0.9 + 0.1 * uniform());
                    double u[3], len = 0.0;
                    for (int i = 0; i < 3; ++i) {
                        u[i] = 2.0 * uniform() - 1.0;
                        if ((k & 3) == 3) u[i] = f.bhat[i] + 0.1 * u[i];
                        len += u[i] * u[i];
                    }
                    for (double& v : u) v /= sqrt(len);
                    double xm[3] = {0, 0, 0}, um[3] = {u[0], u[1], u[2]}, xs[3] = {0, 0, 0}, us[3] = {u[0], u[1], u[2]};
                    quad xq[3] = {0, 0, 0}, uq[3] = {u[0], u[1], u[2]};
                    const quad Bq[3] = {f.B[0], f.B[1], f.B[2]};
                    const emt::FieldMap map = emt::field_step(f, kq, h, um, n);
                    double s = 0.0;
                    for (int i = 0; i < n; ++i) {
                        double xo[3], uo[3];
                        emt::rk4(f, map, s + h, xm, um, xo, uo);
                        for (int a = 0; a < 3; ++a) {
                            xm[a] = xo[a];
                            um[a] = uo[a];
                        }
                        s += h;
                        stages(kq, f.B, h, xs, us);
                        stages((quad)kq, Bq, (quad)h, xq, uq);
                    }
                    emt::field_end(map, um);
                    e[0].add(xm, xq, radius);
                    e[1].add(um, uq, 1.0);
                    e[2].add(xs, xq, radius);
                    e[3].add(us, uq, 1.0);
                }
                printf("%g %d %d", turn, n, axis);
                for (const Error& v : e) printf(" %.3e %.3e", sqrt(v.sum / tracks), v.most);
                printf("\n");
            }
    return 0;
}
