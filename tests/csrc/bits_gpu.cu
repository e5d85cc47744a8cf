// GPU checks of the field transport's bit-level arithmetic against the native
// operations: the float division by a length near 1 (emt_unit.cuh) with the
// hardware's reciprocal square root estimate, the float -> double conversion,
// the integer -> double conversion, the ceiling and the ordered keys
// (emt_device.cuh).  Each kernel counts what it checked and what differed.
#include <cstdint>
#include <cuda_runtime.h>

#include "../../paper_2203_09467_gb300/csrc/emt_device.cuh"

namespace {

__device__ __forceinline__ uint64_t mix(uint64_t z)
{
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__device__ void tally(unsigned long long* counts, unsigned long long checked, unsigned long long wrong)
{
    if (checked) atomicAdd(&counts[0], checked);
    if (wrong) atomicAdd(&counts[1], wrong);
}

// every s in (0.999, 1.001), per_s random components (2^-60 to 1, some next to 1)
__global__ void k_unit(unsigned lo, unsigned n, int per_s, unsigned long long* counts)
{
    unsigned long long checked = 0, wrong = 0;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float s = __uint_as_float(lo + i);
        const float n0 = sqrtf(s);
        float len, r;
        emt::unit::length(s, len, r);
        ++checked;
        wrong += __float_as_uint(len) != __float_as_uint(n0);
        for (int k = 0; k < per_s; ++k) {
            const uint64_t w = mix(((uint64_t)i << 32) | (unsigned)k);
            const uint32_t sign = (uint32_t)w & 0x80000000u;
            const uint32_t b = (k & 3) == 3 ? 0x3F800000u - (uint32_t)(w % 64u)
                                            : ((uint32_t)w & 0x007FFFFFu) | ((127u - (uint32_t)((w >> 32) % 61u)) << 23);
            const float u = __uint_as_float(sign | b);
            ++checked;
            wrong += __float_as_uint(emt::unit::quotient(u, len, r)) != __float_as_uint(u / n0);
        }
    }
    tally(counts, checked, wrong);
}

// every float
__global__ void k_widen(unsigned long long* counts)
{
    unsigned long long checked = 0, wrong = 0;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < (1ull << 32);
         i += (uint64_t)gridDim.x * blockDim.x) {
        const float x = __uint_as_float((uint32_t)i);
        ++checked;
        wrong += __double_as_longlong(emt::widen(x)) != __double_as_longlong((double)x);
    }
    tally(counts, checked, wrong);
}

// every n in [1, 2^20); ceilings of n / 64, of both neighbours and of random
// values of [0, 2^20); keys of random pairs, half of them close together
__global__ void k_small(unsigned long long* counts)
{
    unsigned long long checked = 0, wrong = 0;
    auto ceiling = [&](double q) {
        const int c = (int)ceil(q);
        ++checked;
        wrong += emt::ceil_count(q) != (c < 1 ? 1 : c);
    };
    for (int n = 1 + blockIdx.x * blockDim.x + threadIdx.x; n < (1 << 20); n += gridDim.x * blockDim.x) {
        ++checked;
        wrong += __double_as_longlong(emt::small_int(n)) != __double_as_longlong((double)n);
        const double q = n / 64.0;
        ceiling(q);
        ceiling(__longlong_as_double(__double_as_longlong(q) - 1));
        ceiling(__longlong_as_double(__double_as_longlong(q) + 1));
        const uint64_t w = mix((uint64_t)n), v = mix(w);
        ceiling(__longlong_as_double((long long)((w & 0xFFFFFFFFFFFFFull) | ((uint64_t)(983 + v % 60) << 52))));
        // finite values of either sign
        const uint64_t m = ~(1ull << 62);
        const double a = __longlong_as_double((long long)(w & m));
        const double b = __longlong_as_double((long long)(((n & 1) ? v : w ^ (v >> (20 + n % 40))) & m));
        const int ka = emt::ord_key(a), kb = emt::ord_key(b);
        ++checked;
        wrong += ka != kb && (ka < kb) != (a < b) && a != b;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ceiling(0.0);
        ceiling(5e-324);
    }
    tally(counts, checked, wrong);
}

}  // namespace

// which: 0 unit division, 1 widen, 2 the rest; counts[2]: checked, wrong
extern "C" int bits_check(int which, unsigned long long* counts)
{
    unsigned long long* d = nullptr;
    if (cudaMalloc(&d, 2 * sizeof *d) != cudaSuccess) return 1;
    bool ok = cudaMemset(d, 0, 2 * sizeof *d) == cudaSuccess;
    // bits of the smallest float above 0.999 and the number of floats up to 1.001
    const unsigned lo = 0x3F7FBE77u + 1u, hi = 0x3F8020C5u;
    if (which == 0)
        k_unit<<<304, 128>>>(lo, hi - lo, 4000, d);
    else if (which == 1)
        k_widen<<<1216, 256>>>(d);
    else
        k_small<<<304, 256>>>(d);
    ok = ok && cudaGetLastError() == cudaSuccess && cudaDeviceSynchronize() == cudaSuccess &&
         cudaMemcpy(counts, d, 2 * sizeof *d, cudaMemcpyDeviceToHost) == cudaSuccess;
    cudaFree(d);
    return ok ? 0 : 1;
}
