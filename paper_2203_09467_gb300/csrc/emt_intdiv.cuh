// emt_intdiv.cuh -- IEEE-754 binary64 division and square root on the
// integer pipe.
//
// GB300 executes FP64 at 2 fused multiply-adds per clock per SM (1/64 of
// its FP32 rate), while its integer units issue 64 operations per clock per
// SM.  A correctly rounded FP64 division built from FP64 multiply-adds
// (reciprocal estimate, Newton steps, remainder correction) occupies the
// narrow FP64 pipe for several instructions; the same quotient can be
// formed exactly from the operands' integer significands.  `div_rn(x, y)`
// returns bit for bit what `x / y` returns (round to nearest even): for
// normal operands with a normal quotient it divides the significands on
// the integer pipe; every other case (zeros, subnormals, infinities, NaNs,
// quotients near the ends of the exponent range) takes the native division.
//
// Method.  With x = A 2^ex, y = B 2^ey and A, B in [2^52, 2^53) (A doubled
// when A < B, so that A / B lies in [1, 2)), the result significand is
// RN(A 2^52 / B).  A quotient of two 53-bit integers is never a midpoint
// between two 53-bit integers (if A 2^53 = (2M + 1) B, the power of two in B
// would have to be at least 2^53), so RN(t) = (floor(2t) + 1) / 2 with
// 2t = A 2^53 / B, and only Q' = floor(A 2^53 / B) is needed:
//   1. R ~ 2^115 / B, never above it: an FP32 reciprocal of B's leading 24
//      bits (relative error < 2^-20.9 even three units off), a Newton step
//      R0 -= R0 (B R0 - 1) on 32-bit words (R1 at most 8 units of 2^-32 below
//      1/b), and one on 64-bit words from the low 64 bits of B R1, which hold
//      its whole distance from 2^84 (R at most 60 units of 2^-63 below:
//      2^-58 from the square of R1's error, the rest truncations).
//   2. Q = floor(A R / 2^62): Q' or Q' - 1 (A < 2^54, so 60 units of R move
//      A R / 2^62 by less than 1/4).
//   3. The exact remainder A 2^53 - Q B (in [0, 2B), so its low 64 bits are
//      the whole value) says which.
//
// `sqrt_rn(x)` does the same for the square root: with x = N 2^(2k - 52),
// N in [2^52, 2^54), the result significand is RN(sqrt(N 2^52)), never a
// midpoint (its square would need more than 54 significant bits), so
// Q' = floor(sqrt(N 2^54)) suffices; Y ~ 2^63 / sqrt(N 2^-52), never above it,
// from an FP32 reciprocal square root and two Newton steps
// Y -= Y (N Y^2 2^-178 - 1) / 2 on 32-bit and 64-bit words (Y at most 210
// units low), Q = floor(N Y / 2^62) is Q' or Q' - 1, settled by the exact
// remainder N 2^54 - Q^2 (in [0, 4Q + 4)).
//
// 32-bit words in the first Newton step and one-sided errors (one
// correction instead of two) in place of 128-bit products throughout:
// 10,000-event calorimeter in FP64 46.5 -> 42.8 ms, one event 4.28 -> 4.01 ms
// (36.8 and 3.20 ms with everything else the kernels have changed since).
//
// The FP32 reciprocal (square root) estimates are the only floating-point
// steps; their exact values do not matter, only their error bounds.  Host
// builds (the CPU test of this file) use correctly rounded FP32 results in
// their place, moved by up to three units of the last place to cover the
// hardware estimates' errors.
#pragma once

#include <stdint.h>
#include <math.h>
#include <string.h>

#if defined(__CUDACC__)
#define EMT_HD __host__ __device__ __forceinline__
// one out-of-line copy per kernel: the integer sequences are long, and
// inlined at every call site they overflowed the instruction cache of the
// step kernels (measured on GB300: the calorimeter 20% slower inlined)
#define EMT_HD_CALL static __host__ __device__ __noinline__
#else
#define EMT_HD static inline
#define EMT_HD_CALL static inline
#endif

namespace emt {
namespace intdiv {

EMT_HD uint64_t dbits(double x)
{
    uint64_t b;
    memcpy(&b, &x, 8);
    return b;
}
EMT_HD double bitsd(uint64_t b)
{
    double x;
    memcpy(&x, &b, 8);
    return x;
}

// 32 x 32-bit products: 64-bit, and the high words
EMT_HD uint64_t wide(uint32_t a, uint32_t b) { return (uint64_t)a * b; }
EMT_HD uint32_t mulhi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
EMT_HD int64_t swide(int32_t a, int32_t b) { return (int64_t)a * b; }
EMT_HD int32_t smulhi(int32_t a, int32_t b) { return (int32_t)(((int64_t)a * b) >> 32); }

// floor(a b / 2^62) for a b < 2^126
EMT_HD uint64_t mul_shift62(uint64_t a, uint64_t b)
{
    const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
    const uint64_t t = wide(al, bh) + mulhi(al, bl);
    const uint64_t u = wide(ah, bl) + (uint32_t)t;
    const uint64_t hi = wide(ah, bh) + (uint32_t)(t >> 32) + (uint32_t)(u >> 32);
    return (hi << 2) | ((uint32_t)u >> 30);
}

// FP32 reciprocal (or reciprocal square root) of b in [1, 4) as an integer
// in units of 2^-32, clamped to [1/2, 1): relative error below 2^-22
template <bool kSqrt = false>
EMT_HD uint32_t rcp_q32(float b)
{
#if defined(__CUDA_ARCH__)
    float r;
    if (kSqrt)
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(b));
    else
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(b));
#else
    float r = kSqrt ? 1.0f / sqrtf(b) : 1.0f / b;
#endif
    uint32_t k;
    memcpy(&k, &r, 4);
#if defined(EMT_INTDIV_SEED_ERROR) && !defined(__CUDA_ARCH__)
    k += (uint32_t)EMT_INTDIV_SEED_ERROR(k);  // host test builds: a seed off by a few units
#endif
    k = k < 0x3F000000u ? 0x3F000000u : k;  // [1/2, 1)
    k = k > 0x3F7FFFFFu ? 0x3F7FFFFFu : k;
    return (k << 8) | 0x80000000u;
}

// R ~ 2^115 / B for an integer significand B in [2^52, 2^53); R <= 2^115 / B
EMT_HD uint64_t recip115(uint64_t B)
{
    const uint32_t bb = 0x3F800000u | (uint32_t)((B >> 29) & 0x7FFFFFu);  // B's leading 24 bits, in [1, 2)
    float bf;
    memcpy(&bf, &bb, 4);
    const uint32_t R0 = rcp_q32(bf);
    // e = b R0 - 1 in units of 2^-63, then of 2^-51 (|e| < 2^-20.5)
    const int32_t e = (int32_t)((int64_t)(wide((uint32_t)(B >> 21), R0) ^ (1ull << 63)) >> 12);
    const uint32_t R1 = R0 - 4u - (uint32_t)(smulhi((int32_t)(R0 >> 1), e) >> 18);
    // v = B R1 - 2^84 (|v| < 2^56), then in units of 2^-59
    const int64_t v = (int64_t)(wide((uint32_t)B, R1) + ((uint64_t)((uint32_t)(B >> 32) * R1) << 32));
    const int32_t f = (int32_t)(v >> 25);
    return ((uint64_t)R1 << 31) - 24u - (uint64_t)(swide((int32_t)(R1 >> 1), f) >> 27);
}

// A divisor prepared once for several quotients (its reciprocal R).
struct Divisor {
    double y;
    uint64_t B, R;
    int ey;
};

EMT_HD Divisor divisor(double y)
{
    const uint64_t hy = dbits(y);
    Divisor d;
    d.y = y;
    d.ey = (int)((hy >> 52) & 0x7FF);
    d.B = (hy & ((1ull << 52) - 1)) | (1ull << 52);
    d.R = recip115(d.B);
    return d;
}

// x / d.y, correctly rounded (bit-identical to the IEEE division)
EMT_HD double div_rn(double x, const Divisor& d)
{
    const uint64_t hx = dbits(x);
    const int ex = (int)((hx >> 52) & 0x7FF);
    int er = ex - d.ey + 1023;
    // normal operands and a biased result exponent in [2, 2045] (so that
    // the halving of step 0 and the carry of the rounding stay normal)
    if ((unsigned)(ex - 1) >= 2046u || (unsigned)(d.ey - 1) >= 2046u || (unsigned)(er - 2) >= 2044u) return x / d.y;
    uint64_t A = (hx & ((1ull << 52) - 1)) | (1ull << 52);
    if (A < d.B) {
        A <<= 1;
        er -= 1;
    }
    uint64_t Q = mul_shift62(A, d.R);
    Q += (A << 53) - Q * d.B >= d.B ? 2 : 1;
    Q >>= 1;  // in [2^52, 2^53]; 2^53 carries into the exponent below
    return bitsd(((hx ^ dbits(d.y)) & (1ull << 63)) | (((uint64_t)(er - 1) << 52) + Q));
}

// x / y, correctly rounded (bit-identical to the IEEE division)
EMT_HD_CALL double div_rn(double x, double y) { return div_rn(x, divisor(y)); }

// sqrt(x), correctly rounded (bit-identical to the IEEE square root)
EMT_HD_CALL double sqrt_rn(double x)
{
    const uint64_t hx = dbits(x);
    const int bexp = (int)(hx >> 52);  // sign bit included: negative x takes the native path
    if ((unsigned)(bexp - 1) >= 2046u) return sqrt(x);
    const int odd = (bexp - 1023) & 1;
    const uint64_t N = ((hx & ((1ull << 52) - 1)) | (1ull << 52)) << odd;  // in [2^52, 2^54)
    const int half_e = (bexp - 1023 - odd) / 2;
    // FP32 seed: N 2^-52 in [1, 4) from N's leading 24 bits
    const int top = (int)(N >> 53);  // 1 when N >= 2^53
    const uint32_t nb = ((uint32_t)(127 + top) << 23) | (uint32_t)((N >> (29 + top)) & 0x7FFFFFu);
    float nf;
    memcpy(&nf, &nb, 4);
    const uint32_t Y0 = rcp_q32<true>(nf);
    // e = n y^2 - 1 in units of 2^-62, then of 2^-50 (|e| < 2^-19.5)
    const int32_t e = (int32_t)((int64_t)(wide((uint32_t)(N >> 22), mulhi(Y0, Y0)) - (1ull << 62)) >> 12);
    const uint32_t Y1 = Y0 - 6u - (uint32_t)(smulhi((int32_t)(Y0 >> 1), e) >> 18);
    // w = n Y1^2 - 1 in units of 2^-84 (|w| < 2^57), then of 2^-58
    const uint64_t S = wide(Y1, Y1);
    const uint32_t sl = (uint32_t)S, sh = (uint32_t)(S >> 32), nl = (uint32_t)N, nh = (uint32_t)(N >> 32);
    const int64_t w = (int64_t)(wide(nl, sh) + wide(nh, sl) + mulhi(nl, sl) + ((uint64_t)(nh * sh) << 32));
    const int32_t f = (int32_t)(w >> 26);
    const uint64_t Y = ((uint64_t)Y1 << 31) - 24u - (uint64_t)(swide((int32_t)(Y1 >> 1), f) >> 27);
    // floor(sqrt(N 2^54)) or one less = floor(N y 2^-9)
    uint64_t Q = mul_shift62(N, Y);
    Q += (N << 54) - Q * Q > 2 * Q ? 2 : 1;
    Q >>= 1;  // in [2^52, 2^53]
    return bitsd(((uint64_t)(half_e + 1022) << 52) + Q);
}

}  // namespace intdiv
}  // namespace emt
