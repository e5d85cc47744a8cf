// emt_launch.cuh -- host launchers of the step-loop kernels, instantiated
// once per precision in its own translation unit (different FMA flags).
#pragma once

#include <type_traits>

#include "emt_internal.h"
#include "emt_step.cuh"

namespace emt {

template <int V>
using Int = std::integral_constant<int, V>;
template <bool V>
using Bool = std::integral_constant<bool, V>;

// Calls fn(geometry, field, options) with the kernel instantiation's
// template arguments as constants: the geometry kind, whether a field is on,
// and whether the physics options (multiple scattering, angular
// distributions, Rayleigh) may be on.
template <typename Fn>
static cudaError_t with_variant(bool cylinders, bool field, bool options, Fn fn)
{
    auto with_options = [&](auto g, auto f) { return options ? fn(g, f, Bool<true>{}) : fn(g, f, Bool<false>{}); };
    auto with_field = [&](auto g) { return field ? with_options(g, Bool<true>{}) : with_options(g, Bool<false>{}); };
    return cylinders ? with_field(Int<kGeomCylinders>{}) : with_field(Int<kGeomLayers>{});
}

template <typename R, typename Fn>
static cudaError_t with_variant(const Params<R>& p, Fn fn)
{
    return with_variant(p.geom == kGeomCylinders, p.has_field != 0,
                        (p.mask & (kProcMsc | kProcAngular | kProcRayleigh)) != 0u, fn);
}

// calls fn(block size) for the supported sizes
template <typename Fn>
static cudaError_t with_block(int block, Fn fn)
{
    if (block == 128) return fn(Int<128>{});
    if (block == 256) return fn(Int<256>{});
    return cudaErrorInvalidValue;
}

// Smallest number of resident blocks per SM over the geometry kinds and
// options, with or without a field; kernel(geometry, field, options) names
// the instantiation.  0 on failure.
template <typename Fn>
static int min_blocks(int block, bool field, Fn kernel)
{
    int least = 1 << 30;
    for (int k = 0; k < 4; ++k) {
        int n = 0;
        const cudaError_t e = with_variant((k & 1) != 0, field, (k & 2) != 0, [&](auto g, auto f, auto x) {
            return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel(g, f, x), block, 0);
        });
        if (e != cudaSuccess) return 0;
        if (n < least) least = n;
    }
    return least;
}

template <typename R>
cudaError_t Launch<R>::step(const Params<R>& p, int side, int cin, int cout, int cclr, int grid, int block,
                            cudaStream_t st)
{
    return with_block(block, [&](auto bs) {
        return with_variant(p, [&](auto g, auto f, auto x) {
            k_step<R, bs.value, g.value, f.value, x.value><<<grid, bs.value, 0, st>>>(p, side, cin, cout, cclr);
            return cudaGetLastError();
        });
    });
}

template <typename R>
int Launch<R>::max_blocks_per_sm(int block, bool field)
{
    int n = 0;
    with_block(block, [&](auto bs) {
        n = min_blocks(bs.value, field,
                       [](auto g, auto f, auto x) { return k_step<R, decltype(bs)::value, g.value, f.value, x.value>; });
        return cudaSuccess;
    });
    return n > 0 ? n : 1;
}

template <typename R>
cudaError_t Launch<R>::persist(const Params<R>& p, long long it0, int max_steps, GridSync* gs,
                               long long limit_cycles, int grid, int block, cudaStream_t st)
{
    Params<R> pc = p;
    void* args[] = {&pc, &it0, &max_steps, &gs, &limit_cycles};
    return with_block(block, [&](auto bs) {
        return with_variant(p, [&](auto g, auto f, auto x) {
            return cudaLaunchCooperativeKernel((const void*)k_persist<R, bs.value, g.value, f.value, x.value>,
                                               dim3(grid), dim3(bs.value), args, 0, st);
        });
    });
}

// every block of a cooperative launch must be resident
template <typename R>
int Launch<R>::persist_blocks_per_sm(int block, bool field)
{
    int n = 0;
    with_block(block, [&](auto bs) {
        n = min_blocks(bs.value, field, [](auto g, auto f, auto x) {
            return k_persist<R, decltype(bs)::value, g.value, f.value, x.value>;
        });
        return cudaSuccess;
    });
    return n;
}

template <typename R>
cudaError_t Launch<R>::admit(const Params<R>& p, int side, int cs, int n, const int32_t* ev, const int32_t* type,
                             const double* T, const double* pos, const double* dir, const uint32_t* slot_of_event,
                             const uint32_t* uid_of, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    k_admit<R><<<(n + 255) / 256, 256, 0, st>>>(p, side, cs, n, ev, type, T, pos, dir, slot_of_event, uid_of);
    return cudaGetLastError();
}

template <typename R>
cudaError_t Launch<R>::unspill(const Params<R>& p, int side, int cs, int n, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    k_unspill<R><<<(n + 255) / 256, 256, 0, st>>>(p, side, cs, n);
    return cudaGetLastError();
}

template <typename R>
cudaError_t Launch<R>::set_tracks(const Params<R>& p, int side, int cs, int n, const double* rec,
                                  const uint64_t* uid, const int32_t* slot, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    k_set_tracks<R><<<(n + 255) / 256, 256, 0, st>>>(p, side, cs, n, rec, uid, slot);
    return cudaGetLastError();
}

template <typename R>
cudaError_t Launch<R>::get_tracks(const Params<R>& p, int side, int nG, int nC, double* rec, uint64_t* uid,
                                  int32_t* slot, cudaStream_t st)
{
    int n = nG + nC;
    if (n <= 0) return cudaSuccess;
    k_get_tracks<R><<<(n + 255) / 256, 256, 0, st>>>(p, side, nG, nC, rec, uid, slot);
    return cudaGetLastError();
}

}  // namespace emt

#include "emt_split.cuh"

namespace emt {

// charged tracks of a step in a field sorted by expected substep count (the
// transport kernels take them in that order)
template <typename R>
static void launch_sort(const Params<R>& p, int side, int cin, int grid, cudaStream_t st)
{
    k_sort_keys<R><<<grid, 256, 0, st>>>(p, side, cin);
    k_sort_order<R><<<grid, 256, 0, st>>>(p, cin);
}

template <typename R, bool S>
static cudaError_t launch_split(const Params<R>& p, int side, int cin, int cout, int cclr, int grid_a, int grid_b,
                                int block, cudaStream_t st)
{
    return with_block(block, [&](auto bs) {
        return with_variant(p, [&](auto g, auto f, auto x) {
            if (f.value) launch_sort(p, side, cin, grid_b, st);
            k_transport<R, bs.value, g.value, f.value, S, x.value>
                <<<grid_a, bs.value, 0, st>>>(p, side, cin, cout, cclr);
            k_interact<R, bs.value, S, x.value><<<grid_b, bs.value, 0, st>>>(p, side, cin, cout);
            return cudaGetLastError();
        });
    });
}

template <typename R>
cudaError_t Launch<R>::step_split(const Params<R>& p, int side, int cin, int cout, int cclr, int grid_a, int grid_b,
                                  int block, cudaStream_t st)
{
    return p.max_active > 0 ? launch_split<R, true>(p, side, cin, cout, cclr, grid_a, grid_b, block, st)
                            : launch_split<R, false>(p, side, cin, cout, cclr, grid_a, grid_b, block, st);
}

// resident blocks per SM of the split kernels, with or without track selection
template <typename R>
int Launch<R>::max_blocks_transport(int block, bool field, bool select)
{
    int n = 0;
    with_block(block, [&](auto bs) {
        constexpr int kBs = decltype(bs)::value;
        n = select ? min_blocks(kBs, field, [](auto g, auto f, auto x) {
                         return k_transport<R, kBs, g.value, f.value, true, x.value>;
                     })
                   : min_blocks(kBs, field, [](auto g, auto f, auto x) {
                         return k_transport<R, kBs, g.value, f.value, false, x.value>;
                     });
        return cudaSuccess;
    });
    return n > 0 ? n : 1;
}

template <typename R>
int Launch<R>::max_blocks_interact(int block, bool select)
{
    int n = 0;
    with_block(block, [&](auto bs) {
        constexpr int kBs = decltype(bs)::value;
        n = select ? min_blocks(kBs, false, [](auto, auto, auto x) { return k_interact<R, kBs, true, x.value>; })
                   : min_blocks(kBs, false, [](auto, auto, auto x) { return k_interact<R, kBs, false, x.value>; });
        return cudaSuccess;
    });
    return n > 0 ? n : 1;
}

template <typename R>
cudaError_t Launch<R>::step_pipe(const Params<R>& p, int side, int cin, int cout, int cclr, int grid, int grid_sort,
                                 int block, cudaStream_t st)
{
    return with_block(block, [&](auto bs) {
        return with_variant(p, [&](auto g, auto f, auto x) {
            if (f.value) launch_sort(p, side, cin, grid_sort, st);
            k_pipe<R, bs.value, g.value, f.value, x.value><<<grid, bs.value, 0, st>>>(p, side, cin, cout, cclr);
            return cudaGetLastError();
        });
    });
}

template <typename R>
int Launch<R>::max_blocks_pipe(int block, bool field)
{
    int n = 0;
    with_block(block, [&](auto bs) {
        n = min_blocks(bs.value, field,
                       [](auto g, auto f, auto x) { return k_pipe<R, decltype(bs)::value, g.value, f.value, x.value>; });
        return cudaSuccess;
    });
    return n > 0 ? n : 1;
}

}  // namespace emt

// Explicit instantiations, split across translation units so that the
// heavy kernel families compile in parallel.
#define EMT_INSTANTIATE_FUSED(R)                                                                                    \
    template cudaError_t Launch<R>::step(const Params<R>&, int, int, int, int, int, int, cudaStream_t);           \
    template cudaError_t Launch<R>::admit(const Params<R>&, int, int, int, const int32_t*, const int32_t*,         \
                                          const double*, const double*, const double*, const uint32_t*,         \
                                          const uint32_t*, cudaStream_t);                                         \
    template cudaError_t Launch<R>::set_tracks(const Params<R>&, int, int, int, const double*, const uint64_t*,   \
                                               const int32_t*, cudaStream_t);                                     \
    template cudaError_t Launch<R>::get_tracks(const Params<R>&, int, int, int, double*, uint64_t*, int32_t*,     \
                                               cudaStream_t);                                                     \
    template int Launch<R>::max_blocks_per_sm(int, bool);                                                               \
    template cudaError_t Launch<R>::unspill(const Params<R>&, int, int, int, cudaStream_t);
#define EMT_INSTANTIATE_PERSIST(R)                                                                                  \
    template cudaError_t Launch<R>::persist(const Params<R>&, long long, int, GridSync*, long long, int, int,     \
                                            cudaStream_t);                                                        \
    template int Launch<R>::persist_blocks_per_sm(int, bool);
#define EMT_INSTANTIATE_SPLIT(R)                                                                                    \
    template cudaError_t Launch<R>::step_split(const Params<R>&, int, int, int, int, int, int, int, cudaStream_t); \
    template int Launch<R>::max_blocks_transport(int, bool, bool);                                                 \
    template int Launch<R>::max_blocks_interact(int, bool);
#define EMT_INSTANTIATE_PIPE(R)                                                                                     \
    template cudaError_t Launch<R>::step_pipe(const Params<R>&, int, int, int, int, int, int, int, cudaStream_t);  \
    template int Launch<R>::max_blocks_pipe(int, bool);
