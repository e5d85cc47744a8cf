// emt_field.cuh -- one substep of the FP64 field propagation as a linear map.
//
// P (the kernels' Params, or any type in host code) has the field: baxis (the
// axis of a field along one coordinate axis, else -1), B[3], bmag = |B| and
// bhat[3] = B / |B|.
#pragma once

#include <math.h>

#include "emt_intdiv.cuh"

#if defined(__CUDACC__)
#define EMT_FLD __host__ __device__ __forceinline__
#else
#define EMT_FLD static inline
#endif

namespace emt {

// FP64.  In a uniform field the derivative is linear in u and constant, so
// the four stages of a substep of length h collapse, in exact arithmetic, to
// their stability polynomials: with b = B / |B|, t = kq |B| h, w1 = u x b and
// w2 = w1 x b (and w2 x b = -w1),
//   u' = u + (t - t^3/6) w1 + (t^2/2 - t^4/24) w2
//   x' = x + h u + h (t/2 - t^3/24) w1 + h t^2/6 w2.
// The length of u' follows too: |u'|^2 = 1 + e, e = g |w1|^2 with
// g = t^8/576 - t^6/72 (about 1e-12 in a detector), so u' / |u'| = u' + c u'
// with c = -e/2, and the renormalisation goes into the coefficients, the
// same for all n substeps of the step.  The component along an axis field
// only grows by c of itself, less than a rounding unit: it is formed from the
// path s since the start of the step, u + s (c/h) u, so that the growth is not
// lost substep by substep.  What rounding adds to the length, a unit or so in
// a hundred substeps, is taken off once at the end of the step.
//
// Over n substeps c is not quite constant (|w1|^2 gains g - e of itself in
// each) and the axis component grows by (1 + c)^n: what this leaves out of the
// direction is of the size n^2 e g / 4, below 2^-54 for n |g| < 2^-26: turns t
// below 0.045 at 100 substeps, 0.07 at 8 (the default miss distance and cut
// give t < 0.02 in 2 T).  Larger turns, and a u that does not
// have unit length to start with, are renormalised after each substep; there
// the rounding of t and of the coefficients, the same in every substep, would
// be a phase error that grows with n, so the two turning coefficients are
// formed with what it lost.
//
// The coefficients belong to the length, so a step of n equal substeps forms
// them once; a substep is then 14 FP64 operations along a coordinate axis
// and 33 for any field direction, three deep, against 72 with a square root
// and three divisions stage by stage.  Error against 128-bit arithmetic,
// 4,000 tracks of 1-100 substeps in 2 T: position 1.8e-14 cm rms, direction 1.0e-16;
// stage by stage 1.8e-14 and 2.2e-16; over turns of 0.002 to 0.5 the rms error
// of the map is at most 1.25 times the stages', mostly below it
// (tests/test_field_map.py).  Calorimeter in 2 T, 4,000 events: 2.36 times as
// fast with the map and an explicit renormalisation per substep as stage by
// stage, and 1.12 times again like this with the 32-bit chord test; 109.5 ms now.
struct FieldMap {
    double h;        // displacement along u
    double hp;       // h (1 - t^2/6): along u, components across the field
    double x1, x2;   // displacement along w1, w2
    double c;        // u' / |u'| = u' + c u'
    double u1, u2;   // turn along w1, w2 (with the factor 1 + c)
    double ua, sa;   // axis field: u along the axis at the start, its growth per path
    bool renormalise;  // after every substep
};

// whether n |g| < 2^-26, with n > 1 rounded up to a power of two (exponent
// arithmetic: no instruction on the FP64 pipe)
EMT_FLD bool constant_loss(double g, int n)
{
#if defined(__CUDA_ARCH__)
    const int log2_n = 32 - __clz(n - 1);
#else
    const int log2_n = 32 - __builtin_clz((unsigned)(n - 1));
#endif
    return ((int)(intdiv::dbits(g) >> 32) & 0x7FFFFFFF) + (log2_n << 20) < ((1023 - 26) << 20);
}

// n: substeps of this length (after the last one field_end takes care of the length)
template <typename P>
EMT_FLD FieldMap field_step(const P& p, double kq, double h, const double* u, int n)
{
    FieldMap f;
    const double b = p.baxis >= 0 ? p.B[p.baxis] : p.bmag;
    const double k = kq * b;
    const double t = k * h;
    const double tt = t * t;
    f.h = h;
    f.x2 = h * (tt * (1.0 / 6.0));
    f.hp = h - f.x2;
    f.x1 = h * (t * fma(tt, -1.0 / 24.0, 0.5));
    f.u1 = t * fma(tt, -1.0 / 6.0, 1.0);
    f.u2 = tt * fma(tt, -1.0 / 24.0, 0.5);
    f.ua = p.baxis <= 0 ? u[0] : (p.baxis == 1 ? u[1] : u[2]);
    f.c = 0.0;
    f.sa = 0.0;
    f.renormalise = false;
    if (n > 1) {
        // w = -|w1|^2 / 2 with |w1|^2 = |u|^2 - (u b)^2; g = g_tt t^2
        const double uu = fma(u[0], u[0], fma(u[1], u[1], u[2] * u[2]));
        const double ub =
            p.baxis < 0 ? fma(u[0], p.bhat[0], fma(u[1], p.bhat[1], u[2] * p.bhat[2])) : f.ua;
        const double w = -0.5 * fma(-ub, ub, uu);
        const double g_tt = tt * tt * fma(tt, 1.0 / 576.0, -1.0 / 72.0);
        const double g = g_tt * tt;
        f.renormalise = !(constant_loss(g, n) && fabs(uu - 1.0) < 0x1p-48);
        if (!f.renormalise) {
            f.c = w * g;
            f.sa = w * g_tt * (t * k) * ub;
            f.u1 = fma(f.c, f.u1, f.u1);
            f.u2 = fma(-f.c, 1.0 - f.u2, f.u2);  // along -w2: u' + c u' = u - (u2 - c (1 - u2)) u + ...
        } else {
            // k = kq |B| and t = k h with the parts that their products lost
            // (in any direction also bhat's, along the field: B = bmag bhat + r)
            double lost = 0.0;
            if (p.baxis < 0)
                for (int i = 0; i < 3; ++i) lost = fma(fma(-p.bmag, p.bhat[i], p.B[i]), p.bhat[i], lost);
            const double k_lo = fma(kq, lost, fma(kq, b, -k));
            const double t_lo = fma(k_lo, h, fma(k, h, -t));
            const double tt_lo = fma(2.0 * t, t_lo, fma(t, t, -tt));
            f.u1 = t + fma(t * tt, -1.0 / 6.0, t_lo);
            f.u2 = fma(0.5, tt, fma(tt * tt, -1.0 / 24.0, 0.5 * tt_lo));
        }
    }
    return f;
}

// field along axis A (its sign is in the coefficients): w1 = (0, u_k, -u_j),
// w2 = -(0, u_j, u_k) in the cyclic order A, j, k
template <int A>
EMT_FLD void field_map_axis(const FieldMap& f, double s, const double x[3], const double u[3],
                                               double xo[3], double uo[3])
{
    constexpr int J = (A + 1) % 3, K = (A + 2) % 3;
    xo[A] = fma(f.h, u[A], x[A]);
    xo[J] = x[J] + fma(f.x1, u[K], f.hp * u[J]);
    xo[K] = x[K] + fma(-f.x1, u[J], f.hp * u[K]);
    uo[A] = f.renormalise ? u[A] : fma(s, f.sa, f.ua);
    uo[J] = u[J] + fma(-f.u2, u[J], f.u1 * u[K]);
    uo[K] = u[K] - fma(f.u2, u[K], f.u1 * u[J]);
}

// u / |u|: for a length within 2^-28 of 1 one fused multiply-add per
// component, (1 + e)^(-1/2) being 1 - e/2 to within 2^-54.4
EMT_FLD void renormalise(double u[3])
{
    const double n2 = fma(u[0], u[0], fma(u[1], u[1], u[2] * u[2]));
    const double e = n2 - 1.0;
    if (((int)(intdiv::dbits(e) >> 32) & 0x7FFFFFFF) < ((1023 - 27) << 20)) {
        const double c = -0.5 * e;
#pragma unroll
        for (int i = 0; i < 3; ++i) u[i] = fma(u[i], c, u[i]);
    } else {
        const intdiv::Divisor nd = intdiv::divisor(intdiv::sqrt_rn(n2));
#pragma unroll
        for (int i = 0; i < 3; ++i) u[i] = intdiv::div_rn(u[i], nd);
    }
}

// s: the path from the start of the step (of the map's u) to this substep's end
template <typename P>
EMT_FLD void rk4(const P& p, const FieldMap& f, double s, const double x[3],
                                    const double u[3], double xo[3], double uo[3])
{
    switch (p.baxis) {
    case 0: field_map_axis<0>(f, s, x, u, xo, uo); break;
    case 1: field_map_axis<1>(f, s, x, u, xo, uo); break;
    case 2: field_map_axis<2>(f, s, x, u, xo, uo); break;
    default: {
        // w2 = (u b) b - u splits u' into parts along u, w1 and b w; formed
        // as two cross products, which keep their size small against u
        const double* b = p.bhat;
        double w[3], v[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) w[i] = fma(u[(i + 1) % 3], b[(i + 2) % 3], -(u[(i + 2) % 3] * b[(i + 1) % 3]));
#pragma unroll
        for (int i = 0; i < 3; ++i) v[i] = fma(w[(i + 1) % 3], b[(i + 2) % 3], -(w[(i + 2) % 3] * b[(i + 1) % 3]));
        // along w2 the factor is u2 (1 + c): u2 here is u2 - c (1 - u2), so u2 + c
        const double u2 = f.u2 + f.c;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            xo[i] = x[i] + fma(f.x2, v[i], fma(f.x1, w[i], f.h * u[i]));
            uo[i] = u[i] + fma(u2, v[i], fma(f.u1, w[i], f.c * u[i]));
        }
    }
    }
    if (f.renormalise) renormalise(uo);
}

// the end of a step: take off what rounding added to the length
EMT_FLD void field_end(const FieldMap&, double u[3]) { renormalise(u); }

}  // namespace emt
