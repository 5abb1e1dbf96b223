// d2q9.cu -- launch wrappers of the D2Q9 kernels (d2q9.cuh) for every
// storage format, and the FP64 moments of gathered D2Q9 populations.
#include "d2q9.cuh"
#include "d2q9_diag.cuh"

namespace flb {
namespace d2 {

namespace {

int grid_for(int64_t n, int threads)
{
    int64_t g = (n + threads - 1) / threads;
    if (g > 4096) g = 4096;
    return g < 1 ? 1 : (int)g;
}

// When a step of the one-site kernel lets the next one start, as start_point below:
// at the start in boxes of up to half a block per SM and of many waves, whose blocks
// do not crowd onto few SMs; in between after the loads, or before the stores where
// the in-place steps and the stochastic format, with more to do between the two, would
// still crowd; FP64, whose unit is the bound, before the stores.  us per step, unchained
// / at the start / after the loads / before the stores, plain launches (graphs):
//   FP64 AB   51 x 301 (76 blocks)   10.27 / 17.78 /  8.31 /  8.61   (9.04 / 8.65 / 8.43 / 8.63)
//             117 x 300 (150)        10.56 / 26.37 /  8.41 /  8.66   (9.24 / 13.2 / 8.62 / 8.65)
//             301 x 301 (453)        24.62 / 29.42 / 29.37 / 22.64   (23.2 / 28.9 / 28.9 / 22.8)
//   FP16 AB   301 x 301               5.07 /  4.46 /  2.39 /  2.73   (3.30 / 3.45 / 2.70 / 2.70)
//             401 x 301 (604)         6.18 /  4.01 /  2.85 /  3.36   (3.94 / 3.90 / 3.12 / 3.52)
//             1001 x 601 (2408)      11.91 /  8.80 /  8.76 /  9.23   (9.89 / 8.99 / 8.87 / 9.28)
//   FP16 AA   301 x 301               4.64 /  3.03 /  2.63 /  2.62   (3.10 / 3.11 / 3.03 / 2.67)
//   stochastic AB  301 x 301          6.17 /  5.53 /  3.37 /  3.17   (3.72 / 4.26 / 3.52 / 3.31)
//             117 x 300               4.12 /  2.63 /  2.12 /  2.31   (2.69 / 2.25 / 2.49 / 2.28)
template <class S, int LAYOUT>
StartPoint start_point_one(int64_t blocks, bool in_graph)   // of 256 threads
{
    constexpr int64_t kSMs = 152;
    if (sizeof(S) == 8) return blocks <= kSMs / 2 ? kAfterLoads : kBeforeStores;
    if (blocks <= kSMs) return in_graph || blocks <= kSMs / 2 ? kAtStart : kAfterLoads;
    if (blocks > 6 * kSMs) return kAtStart;
    return LAYOUT == kAB && !Storage<S>::stochastic ? kAfterLoads : kBeforeStores;
}

template <class S, int LAYOUT, bool NOISE, bool FORCE>
cudaError_t step_one(const BoxStep<S> &b, dim3 grid, dim3 block, const uint32_t *p, uint32_t t, cudaStream_t st)
{
    const StartPoint at = start_point_one<S, LAYOUT>((int64_t)grid.x * block.x * block.y / 256, p != nullptr);
    if constexpr (sizeof(S) < 8) {
        if (at == kAtStart)
            return launch_chained(k_stream_collide<S, LAYOUT, NOISE, FORCE, kAtStart>, grid, block, st, b, p, t);
    }
    if (at == kBeforeStores)
        return launch_chained(k_stream_collide<S, LAYOUT, NOISE, FORCE, kBeforeStores>, grid, block, st, b, p, t);
    return launch_chained(k_stream_collide<S, LAYOUT, NOISE, FORCE, kAfterLoads>, grid, block, st, b, p, t);
}

template <class S, int LAYOUT>
cudaError_t step_layout(const BoxStep<S> &b, bool noise, bool force, dim3 grid, dim3 block, const uint32_t *p,
                        uint32_t t, cudaStream_t st)
{
    if (noise && force) return step_one<S, LAYOUT, true, true>(b, grid, block, p, t, st);
    if (noise) return step_one<S, LAYOUT, true, false>(b, grid, block, p, t, st);
    if (force) return step_one<S, LAYOUT, false, true>(b, grid, block, p, t, st);
    return step_one<S, LAYOUT, false, false>(b, grid, block, p, t, st);
}

// V sites per thread: 16-byte accesses for 4-byte formats, 8-byte for 16-bit, V = 2 for FP64.
template <class S>
constexpr int vec_width()
{
    return sizeof(S) == 8 ? 2 : 4;
}

// When a step's blocks let the next step's blocks start.  Any sooner than the SMs
// have room for them without waiting, and they crowd onto the SMs that happen to
// be free, which unbalances every later step; so boxes of about a block per SM
// wait for their loads, and 16-bit boxes of two for their stores.  Beyond that
// 16-bit formats, bound by instructions, start at once, and FP32 waits for its
// stores while the state lies in L2 and for its loads when it streams from HBM
// (the compiler also keeps every load ahead of that point).  us per step, AB,
// unchained / at the start / after the loads / before the stores:
//   FP16  236 x 551 (128 blocks)  4.17 / 4.85 / 2.90 / 2.68; AA in graphs 3.33 / 4.14 / 3.14 / 3.56
//         512 x 512 (256)         6.20 / 5.03 / 4.99 / 3.81
//         1024^2 (1024)           12.35 / 10.12 / 10.18 / 10.16;  3000 x 2400  65.2 / 62.8 / 65.9 / 63.0
//   FP32  236 x 551               6.19 / 6.27 / 3.45 / 3.53
//         752 x 437 (321)         8.24 / 7.37 / 6.39 / 5.47
//         1744 x 864 (1472)       18.49 / 16.08 / 17.10 / 16.24;  3000 x 2400  86.9 / 86.2 / 78.1 / 84.9
// FP64 waits for its loads, but for AB steps without a force of 1.5 to 2 blocks per SM:
// those kernels leave room for three blocks on an SM, so some SMs get three while others
// hold one; the other FP64 kernels leave room for two.
// AA even steps of more than two blocks per SM keep their loads in order: the compiler
// spends six fewer FP64 instructions per thread on them and 76 registers (three blocks
// per SM) instead of 82 (4096 x 2049, even and odd steps 1532 us, 1556 without); below,
// the third block would crowd as above.
//   FP64 AB  256 x 456 (228 blocks)  32.80 / - / 30.23 / 30.16; in graphs 30.75 / - / 30.40 / 31.09
//            256 x 480 (240)         32.80 / - / 44.08 / 30.69; in graphs 30.78 / - / 43.07 / 32.28
//            256 x 600 (300)         32.82 / - / 44.23 / 35.79;  256 x 612 (306)  47.13 / - / 44.26 / 44.00
template <class S, int LAYOUT, bool FORCE>
StartPoint start_point(const BoxStep<S> &b, int64_t blocks, bool in_graph)   // of 256 threads
{
    constexpr int64_t kSMs = 152;
    constexpr int64_t kL2 = 128000000;
    if (sizeof(S) == 8)
        return LAYOUT == kAB && !FORCE && 2 * blocks > 3 * kSMs && blocks <= 2 * kSMs ? kUnchained
               : LAYOUT == kAAEven && blocks > 2 * kSMs                               ? kAfterLoadsInOrder
                                                                                      : kAfterLoads;
    if (sizeof(S) == 2) return blocks <= kSMs ? kAfterLoads : blocks <= 2 * kSMs ? kBeforeStores : kAtStart;
    const bool in_l2 = (LAYOUT == kAB ? 2 : 1) * Q * b.plane * (int64_t)sizeof(S) <= kL2;
    // a graph's launches are close enough for a state in L2: 632 x 640 FP32 takes 5.82 us
    // unchained and 6.93 / 6.22 chained, the boxes of 25,600 to 1.5 M sites at most 3 % less
    if (in_l2 && in_graph) return kUnchained;
    return in_l2 && blocks > 2 * kSMs ? kBeforeStores : kAfterLoads;
}

template <class S, int LAYOUT, bool NOISE, bool FORCE>
cudaError_t step_vec(const BoxStep<S> &b, dim3 grid, dim3 block, const uint32_t *p, uint32_t t, cudaStream_t st)
{
    constexpr int V = vec_width<S>();
    const StartPoint at = start_point<S, LAYOUT, FORCE>(b, (int64_t)grid.x * block.x * block.y / 256, p != nullptr);
    if constexpr (sizeof(S) == 2) {
        if (at == kAtStart)
            return launch_chained(k_stream_collide_vec<S, LAYOUT, NOISE, FORCE, V, kAtStart>, grid, block, st, b, p, t);
    }
    if constexpr (sizeof(S) < 8) {
        if (at == kBeforeStores)
            return launch_chained(k_stream_collide_vec<S, LAYOUT, NOISE, FORCE, V, kBeforeStores>, grid, block, st, b, p, t);
    }
    if constexpr (sizeof(S) == 8 && LAYOUT == kAAEven) {
        if (at == kAfterLoadsInOrder)
            return launch_chained(k_stream_collide_vec<S, LAYOUT, NOISE, FORCE, V, kAfterLoadsInOrder>, grid, block, st, b,
                                  p, t);
    }
    if constexpr (sizeof(S) >= 4) {
        if (at == kUnchained) {
            constexpr int kAny = sizeof(S) == 8 ? kAfterLoads : kBeforeStores;
            k_stream_collide_vec<S, LAYOUT, NOISE, FORCE, V, kAny><<<grid, block, 0, st>>>(b, p, t);
            return cudaGetLastError();
        }
    }
    return launch_chained(k_stream_collide_vec<S, LAYOUT, NOISE, FORCE, V, kAfterLoads>, grid, block, st, b, p, t);
}

template <class S, int LAYOUT>
cudaError_t step_layout_vec(const BoxStep<S> &b, bool noise, bool force, dim3 grid, dim3 block, const uint32_t *p,
                            uint32_t t, cudaStream_t st)
{
    if (noise && force) return step_vec<S, LAYOUT, true, true>(b, grid, block, p, t, st);
    if (noise) return step_vec<S, LAYOUT, true, false>(b, grid, block, p, t, st);
    if (force) return step_vec<S, LAYOUT, false, true>(b, grid, block, p, t, st);
    return step_vec<S, LAYOUT, false, false>(b, grid, block, p, t, st);
}

}  // namespace

template <class S>
cudaError_t launch_step(const BoxStep<S> &b, int layout, bool noise, bool force, int bx, int by, int V,
                        const uint32_t *step_ptr, uint32_t step, cudaStream_t st)
{
    if (V > 1) {
        // vectorised: needs nx % V == 0 and whole warps
        constexpr int W = vec_width<S>();
        const int T = bx * by;
        if (b.nx % W != 0 || T % 32 != 0 || T > 256) return cudaErrorInvalidValue;
        const int64_t items = (int64_t)(b.nx / W) * b.ny;
        const dim3 grid((unsigned)((items + T - 1) / T)), block(bx, by, 1);
        switch (layout) {
        case kAB: return step_layout_vec<S, kAB>(b, noise, force, grid, block, step_ptr, step, st);
        case kAAEven: return step_layout_vec<S, kAAEven>(b, noise, force, grid, block, step_ptr, step, st);
        default: return step_layout_vec<S, kAAOdd>(b, noise, force, grid, block, step_ptr, step, st);
        }
    }
    const int gy = (b.ny + by - 1) / by;
    const int64_t blocks = (int64_t)b.gx * gy;
    if (blocks > 0x7FFFFFFF || bx * by > 256 || bx < 1 || by < 1) return cudaErrorInvalidValue;
    const dim3 grid((unsigned)blocks), block(bx, by, 1);
    switch (layout) {
    case kAB: return step_layout<S, kAB>(b, noise, force, grid, block, step_ptr, step, st);
    case kAAEven: return step_layout<S, kAAEven>(b, noise, force, grid, block, step_ptr, step, st);
    default: return step_layout<S, kAAOdd>(b, noise, force, grid, block, step_ptr, step, st);
    }
}

template <class S>
cudaError_t launch_gather(const S *buf, int64_t plane, int layout, int nx, int ny, int y0, int nyc, double rho0,
                          double *out, cudaStream_t st)
{
    k_gather<S><<<grid_for((int64_t)nx * nyc, 256), 256, 0, st>>>(buf, plane, layout, nx, ny, y0, nyc, rho0, out);
    return cudaGetLastError();
}

template <class S>
cudaError_t launch_gather_sites(const S *buf, int64_t plane, int layout, int nx, int ny, double rho0,
                                const int64_t *sites, int64_t nsites, double *out, cudaStream_t st)
{
    k_gather_sites<S><<<grid_for(nsites, 256), 256, 0, st>>>(buf, plane, layout, nx, ny, rho0, sites, nsites, out);
    return cudaGetLastError();
}

template <class S>
cudaError_t launch_scatter(S *buf, int64_t plane, int layout, int nx, int ny, int y0, int nyc, double rho0,
                           const double *in, cudaStream_t st)
{
    k_scatter<S><<<grid_for((int64_t)nx * nyc, 256), 256, 0, st>>>(buf, plane, layout, nx, ny, y0, nyc, rho0, in);
    return cudaGetLastError();
}

template <class S>
cudaError_t launch_init_equilibrium(S *buf, int64_t plane, int layout, int nx, int ny, int y0, int nyc, double rho0,
                                    const double *u, cudaStream_t st)
{
    k_init_equilibrium<S><<<grid_for((int64_t)nx * nyc, 256), 256, 0, st>>>(buf, plane, layout, nx, ny, y0, nyc,
                                                                           rho0, u);
    return cudaGetLastError();
}

template <class S>
cudaError_t launch_stats_partial(const S *buf, int64_t plane, int layout, int nx, int ny, double rho0,
                                 double *partial, int nblocks, cudaStream_t st)
{
    k_stats_partial<S><<<nblocks, 256, 0, st>>>(buf, plane, layout, nx, ny, rho0, partial);
    return cudaGetLastError();
}

template <class S>
cudaError_t launch_density(const S *buf, int64_t plane, int layout, int nx, int ny, typename Storage<S>::R *field,
                           cudaStream_t st)
{
    k_density<S><<<grid_for((int64_t)nx * ny, 256), 256, 0, st>>>(buf, plane, layout, nx, ny, field);
    return cudaGetLastError();
}

__global__ void k_moments(const double *__restrict__ n, int64_t slab, int nx, int ny, int y0, double force_amp,
                          double *__restrict__ rho, double *__restrict__ j, double *__restrict__ Pi)
{
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < slab; s += (int64_t)gridDim.x * blockDim.x) {
        double r = 0, jx = 0, jy = 0, pxx = 0, pyy = 0, pxy = 0;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const double v = n[i * slab + s];
            const double cx = vel_x(i), cy = vel_y(i);
            r += v;
            jx += v * cx;
            jy += v * cy;
            pxx += v * cx * cx;
            pyy += v * cy * cy;
            pxy += v * cx * cy;
        }
        if (force_amp != 0.0) {
            const int y = y0 + (int)(s / nx);
            jx += 0.5 * force_amp * sinpi(2.0 * y / ny);
        }
        if (rho) rho[s] = r;
        if (j) {
            j[s] = jx;
            j[slab + s] = jy;
        }
        if (Pi) {
            Pi[s] = pxx;
            Pi[slab + s] = pyy;
            Pi[2 * slab + s] = pxy;
        }
    }
}

cudaError_t launch_moments(const double *n, int64_t slab, int nx, int ny, int y0, double force_amp, double *rho,
                           double *j, double *Pi, cudaStream_t st)
{
    k_moments<<<grid_for(slab, 256), 256, 0, st>>>(n, slab, nx, ny, y0, force_amp, rho, j, Pi);
    return cudaGetLastError();
}

#define FLB_D2_INSTANTIATE(S)                                                                                       \
    template cudaError_t launch_step<S>(const BoxStep<S> &, int, bool, bool, int, int, int, const uint32_t *,      \
                                        uint32_t, cudaStream_t);                                                    \
    template cudaError_t launch_gather<S>(const S *, int64_t, int, int, int, int, int, double, double *,           \
                                          cudaStream_t);                                                            \
    template cudaError_t launch_gather_sites<S>(const S *, int64_t, int, int, int, double, const int64_t *,        \
                                                int64_t, double *, cudaStream_t);                                   \
    template cudaError_t launch_scatter<S>(S *, int64_t, int, int, int, int, int, double, const double *,          \
                                           cudaStream_t);                                                           \
    template cudaError_t launch_init_equilibrium<S>(S *, int64_t, int, int, int, int, int, double, const double *, \
                                                    cudaStream_t);                                                  \
    template cudaError_t launch_stats_partial<S>(const S *, int64_t, int, int, int, double, double *, int,         \
                                                 cudaStream_t);                                                     \
    template cudaError_t launch_density<S>(const S *, int64_t, int, int, int, typename Storage<S>::R *, cudaStream_t);

FLB_D2_INSTANTIATE(double)
FLB_D2_INSTANTIATE(float)
FLB_D2_INSTANTIATE(__half)
FLB_D2_INSTANTIATE(__nv_bfloat16)
FLB_D2_INSTANTIATE(bf16sr)

}  // namespace d2
}  // namespace flb
