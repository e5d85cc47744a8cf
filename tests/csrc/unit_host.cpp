// CPU check of emt_unit.cuh against sqrtf and the C division: every s in
// (0.999, 1.001) with the reciprocal square root estimate moved by -2..2 units
// of its last place, and quotients of random components (2^-60 to 1, and next
// to the length) by every n of that range.  Prints checked and wrong counts.
#include <cstdint>
#include <cstdio>
#include <cmath>
#include <cstdlib>
#include <cstring>

static int g_err = 0;
#define EMT_UNIT_SEED_ERROR g_err
#include "../../paper_2203_09467_gb300/csrc/emt_unit.cuh"

static uint64_t g_s = 0x9E3779B97F4A7C15ull;
static uint32_t next()
{
    g_s ^= g_s << 13;
    g_s ^= g_s >> 7;
    g_s ^= g_s << 17;
    return (uint32_t)(g_s >> 32);
}

int main(int argc, char** argv)
{
    const int per_s = argc > 1 ? atoi(argv[1]) : 40;
    long checked = 0, wrong = 0;
    for (float s = nextafterf(0.999f, 2.0f); s < 1.001f; s = nextafterf(s, 2.0f)) {
        const float n0 = sqrtf(s);
        for (g_err = -2; g_err <= 2; ++g_err) {
            float n, r;
            emt::unit::length(s, n, r);
            ++checked;
            if (n != n0) {
                if (wrong++ < 5) printf("sqrt(%a): %a, here %a (estimate off by %d)\n", s, n0, n, g_err);
            }
            for (int k = 0; k < per_s; ++k) {
                const uint32_t w = next();
                // sign, exponent 2^-60 .. 1, 23 random bits; every fourth next to 1
                const int e = (k & 3) == 3 ? 126 : 127 - (int)(next() % 61);
                uint32_t b = (w & 0x807FFFFFu) | ((uint32_t)e << 23);
                if ((k & 3) == 3) b = (w & 0x80000000u) | (0x3F800000u - (w % 64u));
                float u;
                memcpy(&u, &b, 4);
                const float q0 = u / n0, q = emt::unit::quotient(u, n, r);
                ++checked;
                if (q != q0 && wrong++ < 5) printf("%a / %a: %a, here %a (estimate off by %d)\n", u, n0, q0, q, g_err);
            }
        }
    }
    printf("%ld %ld\n", checked, wrong);
    return wrong != 0;
}
