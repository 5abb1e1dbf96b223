// step_impl.cuh -- launch wrappers of the templated kernels; included by the
// step_<format>.cu files, each of which instantiates them for one storage
// format so the formats compile in parallel.
#pragma once

#include "diag_kernels.cuh"
#include "kernels.cuh"

namespace flb {

namespace detail {

template <class S, int LAYOUT, int NOISE, bool FORCE, int V>
cudaError_t step_one(const BoxStep<S> &b, const Launch &L, const uint32_t *step_ptr, uint32_t step, cudaStream_t st)
{
    const int g = b.nx / V, T = L.bx * L.by;
    if constexpr (V > 1) {
        // the three-dimensional grids end at 65535 along y and z; longer boxes take the forms with one grid index
        constexpr int kGridYZ = 65535;
        const bool off32 = (uint64_t)Q * (uint64_t)b.plane < (1ull << 32);
        const bool planes = b.nzl <= kGridYZ, lines = planes && b.ny <= kGridYZ;
        const int warp_blocks = b.ny / L.by + (b.ny % L.by != 0);
        if (L.warprow && planes && warp_blocks <= kGridYZ)
            return launch_chained(k_stream_collide<S, LAYOUT, NOISE, FORCE, V, kWarpRow>, dim3(1, warp_blocks, b.nzl),
                                  dim3(L.bx, L.by), st, b, step_ptr, step);
        if (L.rows == 1 && off32 && lines) {
            const dim3 grid(1, b.ny, b.nzl), block((g + 31) / 32 * 32);
            if (g % 32 == 0)
                return launch_chained(k_stream_collide<S, LAYOUT, NOISE, FORCE, V, kOneRow, true>, grid, block, st, b,
                                      step_ptr, step);
            return launch_chained(k_stream_collide<S, LAYOUT, NOISE, FORCE, V, kRagRow, true>, grid, block, st, b,
                                  step_ptr, step);
        }
        if (L.rows > 0) {
            BoxStep<S> r = b;
            r.rows = L.rows;
            const int64_t nrows = (int64_t)b.ny * b.nzl;
            const dim3 grid((unsigned)((nrows + L.rows - 1) / L.rows)), block((L.rows * g + 31) / 32 * 32);
            return launch_chained(k_stream_collide<S, LAYOUT, NOISE, FORCE, V, kRows>, grid, block, st, r, step_ptr,
                                  step);
        }
        if (L.edgerow && lines)
            return launch_chained(k_stream_collide<S, LAYOUT, NOISE, FORCE, V, kEdgeRow>,
                                  dim3((g + T - 1) / T, b.ny, b.nzl), dim3(T), st, b, step_ptr, step);
    }
    const int64_t items = (int64_t)g * b.ny * b.nzl;
    return launch_chained(k_stream_collide<S, LAYOUT, NOISE, FORCE, V>, dim3((unsigned)((items + T - 1) / T)), dim3(T),
                          st, b, step_ptr, step);
}

template <class S, int LAYOUT, int NOISE, bool FORCE, int V>
cudaError_t step_batch(const BatchParams<S> &P, int total_blocks, const Launch &L, const uint32_t *step_ptr,
                       uint32_t step, cudaStream_t st)
{
    const dim3 block(L.bx * L.by);
    if constexpr (kBatchMinBlocks<S, LAYOUT, V> == 4) {
        // three blocks of 256 threads per SM instead of four (see kBatchMinBlocks)
        bool tiled = sizeof(S) == 4;
        for (int k = 0; k < P.nboxes; ++k) tiled = tiled && P.boxes[k].warprow;
        if (tiled || (int64_t)total_blocks * (int64_t)block.x <= 4 * 152 * 256)
            return launch_chained(k_stream_collide_batch<S, LAYOUT, NOISE, FORCE, V, 3>, dim3(total_blocks), block, st, P,
                                  step_ptr, step);
    }
    return launch_chained(k_stream_collide_batch<S, LAYOUT, NOISE, FORCE, V>, dim3(total_blocks), block, st, P,
                          step_ptr, step);
}

template <class S, int LAYOUT, int NOISE, bool FORCE>
cudaError_t step_v(const BoxStep<S> &b, const Launch &L, const uint32_t *p, uint32_t t, cudaStream_t st)
{
    switch (L.V) {
    case 1: return step_one<S, LAYOUT, NOISE, FORCE, 1>(b, L, p, t, st);
    case 2: return step_one<S, LAYOUT, NOISE, FORCE, 2>(b, L, p, t, st);
    case 4: return step_one<S, LAYOUT, NOISE, FORCE, (sizeof(S) * 4 > 16 ? 2 : 4)>(b, L, p, t, st);
    }
    return cudaErrorInvalidValue;
}

template <class S, int LAYOUT, int NOISE, bool FORCE>
cudaError_t batch_v(const BatchParams<S> &P, int tb, const Launch &L, const uint32_t *p, uint32_t t, cudaStream_t st)
{
    switch (L.V) {
    case 1: return step_batch<S, LAYOUT, NOISE, FORCE, 1>(P, tb, L, p, t, st);
    case 2: return step_batch<S, LAYOUT, NOISE, FORCE, 2>(P, tb, L, p, t, st);
    case 4: return step_batch<S, LAYOUT, NOISE, FORCE, (sizeof(S) * 4 > 16 ? 2 : 4)>(P, tb, L, p, t, st);
    }
    return cudaErrorInvalidValue;
}

template <class S, int LAYOUT>
cudaError_t step_nf(const BoxStep<S> &b, int noise, bool force, const Launch &L, const uint32_t *p, uint32_t t,
                    cudaStream_t st)
{
    if (noise == 2) return force ? step_v<S, LAYOUT, 2, true>(b, L, p, t, st) : step_v<S, LAYOUT, 2, false>(b, L, p, t, st);
    if (noise) return force ? step_v<S, LAYOUT, 1, true>(b, L, p, t, st) : step_v<S, LAYOUT, 1, false>(b, L, p, t, st);
    return force ? step_v<S, LAYOUT, 0, true>(b, L, p, t, st) : step_v<S, LAYOUT, 0, false>(b, L, p, t, st);
}

template <class S, int LAYOUT>
cudaError_t batch_nf(const BatchParams<S> &P, int tb, int noise, bool force, const Launch &L, const uint32_t *p,
                     uint32_t t, cudaStream_t st)
{
    if (noise == 2)
        return force ? batch_v<S, LAYOUT, 2, true>(P, tb, L, p, t, st) : batch_v<S, LAYOUT, 2, false>(P, tb, L, p, t, st);
    if (noise)
        return force ? batch_v<S, LAYOUT, 1, true>(P, tb, L, p, t, st) : batch_v<S, LAYOUT, 1, false>(P, tb, L, p, t, st);
    return force ? batch_v<S, LAYOUT, 0, true>(P, tb, L, p, t, st) : batch_v<S, LAYOUT, 0, false>(P, tb, L, p, t, st);
}

inline int grid_for(int64_t n, int block)
{
    int64_t g = (n + block - 1) / block;
    if (g > 4096) g = 4096;
    if (g < 1) g = 1;
    return (int)g;
}

}  // namespace detail

template <class S>
cudaError_t launch_step(const BoxStep<S> &b, int layout, int noise, bool force, const Launch &L,
                        const uint32_t *step_ptr, uint32_t step, cudaStream_t st)
{
    switch (layout) {
    case kAB: return detail::step_nf<S, kAB>(b, noise, force, L, step_ptr, step, st);
    case kAAEven: return detail::step_nf<S, kAAEven>(b, noise, force, L, step_ptr, step, st);
    case kAAOdd: return detail::step_nf<S, kAAOdd>(b, noise, force, L, step_ptr, step, st);
    }
    return cudaErrorInvalidValue;
}

template <class S>
cudaError_t launch_step_batch(const BatchParams<S> &P, int total_blocks, int layout, int noise, bool force,
                              const Launch &L, const uint32_t *step_ptr, uint32_t step, cudaStream_t st)
{
    switch (layout) {
    case kAB: return detail::batch_nf<S, kAB>(P, total_blocks, noise, force, L, step_ptr, step, st);
    case kAAEven: return detail::batch_nf<S, kAAEven>(P, total_blocks, noise, force, L, step_ptr, step, st);
    case kAAOdd: return detail::batch_nf<S, kAAOdd>(P, total_blocks, noise, force, L, step_ptr, step, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace flb

// The stream-collide kernels of one storage format S and one layout L
// (instantiated in step_<format>_<layout>.cu, so the 15 kernel TUs compile in
// parallel); the dispatching TU declares them extern.
#define FLB_LAYOUT_FUNCS(PREFIX, S, L)                                                                              \
    namespace flb {                                                                                                 \
    namespace detail {                                                                                              \
    PREFIX template cudaError_t step_nf<S, L>(const BoxStep<S> &, int, bool, const Launch &, const uint32_t *,      \
                                              uint32_t, cudaStream_t);                                              \
    PREFIX template cudaError_t batch_nf<S, L>(const BatchParams<S> &, int, int, bool, const Launch &,              \
                                               const uint32_t *, uint32_t, cudaStream_t);                           \
    }                                                                                                               \
    }
#define FLB_INSTANTIATE_LAYOUT(S, L) FLB_LAYOUT_FUNCS(, S, L)

#define FLB_INSTANTIATE(S)                                                                                          \
    FLB_LAYOUT_FUNCS(extern, S, kAB)                                                                                \
    FLB_LAYOUT_FUNCS(extern, S, kAAEven)                                                                            \
    FLB_LAYOUT_FUNCS(extern, S, kAAOdd)                                                                             \
    namespace flb {                                                                                                 \
    template cudaError_t launch_step<S>(const BoxStep<S> &, int, int, bool, const Launch &, const uint32_t *,       \
                                        uint32_t, cudaStream_t);                                                    \
    template cudaError_t launch_step_batch<S>(const BatchParams<S> &, int, int, int, bool, const Launch &,         \
                                              const uint32_t *, uint32_t, cudaStream_t);                            \
    template cudaError_t launch_gather<S>(const S *, int64_t, int, int, int, int, int, int, double, double *,      \
                                          cudaStream_t);                                                            \
    template cudaError_t launch_gather_sites<S>(const S *, int64_t, int, int, int, int, double, const int64_t *,    \
                                                int64_t, double *, cudaStream_t);                                   \
    template cudaError_t launch_scatter<S>(S *, int64_t, int, int, int, int, int, int, double, const double *,     \
                                           cudaStream_t);                                                           \
    template cudaError_t launch_init_equilibrium<S>(S *, int64_t, int, int, int, int, int, int, double,            \
                                                    const double *, cudaStream_t);                                  \
    template cudaError_t launch_stats_partial<S>(const S *, int64_t, int, int, int, int, double, double *, int,    \
                                                 typename Storage<S>::R *, cudaStream_t);                           \
    template cudaError_t launch_stats_partial_batch<S>(const StatsTable<S> &, int, int, cudaStream_t);             \
    }
