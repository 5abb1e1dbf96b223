// profile.cuh -- plane averages of the canonical state (flb_box_z_profile) for
// both lattices.
//
// A unit is a z-plane of a D3Q19 box or a row y of a D2Q9 box.  The shifts of
// a population inside its unit do not change the unit's sum, so the sum of the
// canonical n_i over unit u is the sum of one slot's contiguous unit u - c_i: the
// first kernel sums every unit of every slot as one stream, the second combines
// the Q sums of each unit.  FP32 is bound by HBM: 512^3 1.40 ms per call (10.2 GB at
// 7.3 TB/s), 64^3 27 us, of which about 20 are the call's launches and wait; 16-bit
// formats by the additions (512^3 FP16 1.08 ms, 256^3 bfloat16 0.17).  One block per
// plane with every site's populations added in FP64 took 34.3 ms, 160 us, 34.2 and 4.3 ms.
#pragma once

#include "d3q19.cuh"
#include "internal.h"

namespace flb {
namespace profile {

// a + b without a rounding error: the sum and what it lost (Knuth's TwoSum).
__device__ __forceinline__ float two_sum(float a, float b, float &err)
{
    const float s = __fadd_rn(a, b), t = __fadd_rn(a, -s);   // -t: what s took of b
    err = __fadd_rn(__fadd_rn(a, -__fadd_rn(s, t)), __fadd_rn(b, t));
    return s;
}

// A running sum of 16- or 32-bit values as an unevaluated sum of three floats: an
// FP64 addition occupies an SM quarter's FP64 unit for 64 cycles per warp, and a
// conversion to FP64 as long, thirteen FP32 additions for thirteen.  hi takes the
// values, mid what hi loses, lo what mid loses; settle() passes what has gathered in
// mid and lo upwards.  With n values between two calls mid is at most n 2^-24 of the
// largest hi, and an addition to lo rounds by at most 2^-24 n 2^-24 n 2^-24 of it,
// 2^-61 for n = 40: less than the 2^-53 of an FP64 addition.  A sum that leaves the
// range of FP32 (or meets an infinity or NaN) shows as non-finite; its values are then
// summed again in FP64.
struct TripleSum {
    float hi = 0.f, mid = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float v)
    {
        float e, e2;
        hi = two_sum(hi, v, e);
        mid = two_sum(mid, e, e2);
        lo += e2;
    }
    __device__ __forceinline__ void add(const TripleSum &o)
    {
        float e;
        add(o.hi);
        mid = two_sum(mid, o.mid, e);
        lo += e + o.lo;
    }
    __device__ __forceinline__ void settle()
    {
        float t;
        hi = two_sum(hi, mid, t);
        mid = two_sum(t, lo, lo);
    }
    __device__ __forceinline__ bool finite() const { return isfinite(hi) && isfinite(mid) && isfinite(lo); }
    __device__ __forceinline__ double value() const { return (double)hi + ((double)mid + (double)lo); }
};

constexpr int kThreads = 128;     // per block; 16 blocks per SM (32 registers): 512^3 FP32 1.40 ms, 1.75 with what is left
                                  // free (40); 256 threads take 1.40 ms too, but 64^3 bfloat16 30.6 us against 27.2
constexpr int kUnroll = 4;        // 16-byte loads in flight per thread
template <class S>
constexpr int kSettle = sizeof(S) == 4 ? 8 : 4;   // loads between two calls of settle: 32 values

// The units of one pass: the sums of nsum consecutive units from `first` on (modulo
// the box's units), then the means of n units, of which the first is the lead-th
// sum.  A box of at most kPassUnits units is one pass over all of its sums (lead =
// 0, the neighbours of the ends wrap around); a larger one takes kPassUnits at a
// time with one sum more at either side (lead = 1), so that the scratch stays at
// 4 units + Q nsum doubles (10 MB) and the indices of sums and means within 32 bits.
struct Pass {
    int first, nsum, lead, n;
};
constexpr int kPassUnits = 65536;
__host__ __device__ inline Pass pass_from(int u0, int units)
{
    if (units <= kPassUnits) return Pass{0, units, 0, units};
    const int n = units - u0 < kPassUnits ? units - u0 : kPassUnits;
    return Pass{(u0 ? u0 : units) - 1, n + 2, 1, n};
}
// the box's unit of sum u, and the sum that slot i's unit k of the means comes from
__host__ __device__ inline int unit_of_sum(const Pass &p, int u, int units)
{
    const unsigned v = (unsigned)p.first + (unsigned)u;
    return (int)(v < (unsigned)units ? v : v - (unsigned)units);
}
__host__ __device__ inline int sum_of_mean(const Pass &p, int k, int shift)
{
    const int u = k + p.lead - shift;
    return u < 0 ? u + p.nsum : (u >= p.nsum ? u - p.nsum : u);
}

// T threads (a warp or the block) sum chunk c of `chunks` of sum u (unit
// unit_of_sum) of slot q, M elements per unit, into part[(q nsum + u) chunks + c];
// work item w is (c, q, u) with u fastest.
template <class S, int T>
__global__ void __launch_bounds__(kThreads, 16) k_unit_sums(const S *__restrict__ buf, int64_t plane, int64_t M, int units,
                                                        Pass P, int64_t items, int chunks, double *__restrict__ part)
{
    constexpr int E = 16 / sizeof(S);   // elements per 16-byte load
    constexpr int kWarps = T / 32;
    const int tid = (int)threadIdx.x % T;
    const int64_t w = (int64_t)blockIdx.x * (kThreads / T) + threadIdx.x / T;
    if (w >= items) return;             // whole warps: T is 32 or the block
    const int u = (int)(w % P.nsum);
    const int64_t qc = w / P.nsum;
    const int q = (int)(qc / chunks), c = (int)(qc % chunks);
    const int64_t per = (M + chunks - 1) / chunks, c0 = c * per;
    const int64_t n = max((int64_t)0, min(per, M - c0));
    const S *p = buf + q * plane + unit_of_sum(P, u, units) * M + c0;
    // up to the first 16-byte boundary and behind the last one: single elements
    const int64_t head = min(n, (int64_t)((16 - reinterpret_cast<uintptr_t>(p) % 16) % 16 / sizeof(S)));
    const int64_t vecs = (n - head) / E, tail = n - head - vecs * E;
    const uint4 *v = reinterpret_cast<const uint4 *>(p + head);
    // f(value), and after(loads) after every kUnroll loads
    auto each = [&](auto f, auto after) {
        if (tid < head) f(p[tid]);
        if (tid < tail) f(p[head + vecs * E + tid]);
        int loads = 0;
        for (int64_t i0 = tid; i0 < vecs; i0 += kUnroll * T) {
            uint4 x[kUnroll];
#pragma unroll
            for (int r = 0; r < kUnroll; ++r)
                x[r] = i0 + r * T < vecs ? v[i0 + r * T] : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int r = 0; r < kUnroll; ++r) {
                const S *e = reinterpret_cast<const S *>(&x[r]);
#pragma unroll
                for (int k = 0; k < E; ++k) f(e[k]);
            }
            after(loads += kUnroll);
        }
    };
    auto over_lanes = [](double x) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
        return x;
    };
    double *const to = part + ((int64_t)q * P.nsum + u) * chunks + c;
    if constexpr (sizeof(S) < 8) {
        TripleSum s;
        each([&](S x) { s.add(Storage<S>::load(x)); },
             [&](int loads) {
                 if (loads % kSettle<S> == 0) s.settle();
             });
        // the first warp adds the block's warps lane by lane, then its lanes
        __shared__ float all[3][kWarps][32];
        bool fp64 = !s.finite();
        if constexpr (kWarps > 1) {
            all[0][tid / 32][tid % 32] = s.hi;
            all[1][tid / 32][tid % 32] = s.mid;
            all[2][tid / 32][tid % 32] = s.lo;
            fp64 = __syncthreads_or(fp64);
        }
        if (!__any_sync(0xffffffffu, fp64)) {
            if (tid >= 32) return;
            auto of = [&](int k) { return TripleSum{all[0][k][tid], all[1][k][tid], all[2][k][tid]}; };
#pragma unroll
            for (int k = 1; k < kWarps; ++k) s.add(of(k));
#pragma unroll
            for (int off = 16; off > 0; off >>= 1)
                s.add(TripleSum{__shfl_xor_sync(0xffffffffu, s.hi, off), __shfl_xor_sync(0xffffffffu, s.mid, off),
                                __shfl_xor_sync(0xffffffffu, s.lo, off)});
            const bool ok = !__any_sync(0xffffffffu, !s.finite());   // else out of range only together
            if (kWarps > 1 || ok) {
                double sum = s.value();
                if (!ok) {
                    sum = 0.0;
                    for (int k = 0; k < kWarps; ++k) sum += of(k).value();
                    sum = over_lanes(sum);
                }
                if (tid == 0) *to = sum;
                return;
            }
        }
    }
    double sum = 0.0;
    each([&](S x) { sum += Storage<S>::to_double(x); }, [](int) {});
    sum = over_lanes(sum);
    if constexpr (kWarps > 1) {
        __shared__ double wsum[kWarps];
        if ((tid & 31) == 0) wsum[tid >> 5] = sum;
        __syncthreads();
        sum = 0.0;
        if (tid == 0) {
#pragma unroll
            for (int k = 0; k < kWarps; ++k) sum += wsum[k];
        }
    }
    if (tid == 0) *to = sum;
}

// The unit of a thread of k_unit_means.  Warps are counted, not threads: 2^27 units have
// 2^32 threads.
__host__ __device__ inline int unit_of(unsigned block, unsigned block_threads, unsigned thread)
{
    return (int)(block * (block_threads / 32) + thread / 32);
}

// Warp u, unit u of the pass's n: out[u] = rho0 + sum_i s_i / M, out[n + 3 u + a] =
// sum_i c_ia s_i / M, s_i (lane i) the sum of the deviation n_i over the unit.  D2: the D2Q9 velocities
// in rows y (the third component is 0).
template <bool D2>
__global__ void __launch_bounds__(128) k_unit_means(const double *__restrict__ part, int layout, int64_t M, Pass P,
                                                    int chunks, double rho0, double *__restrict__ out)
{
    constexpr int NQ = D2 ? 9 : 19;
    const int i = (int)threadIdx.x & 31, u = unit_of(blockIdx.x, blockDim.x, threadIdx.x);
    if (u >= P.n) return;   // whole warps
    constexpr int vx[2][19] = {{0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1},
                               {0, 1, -1, 0, 0, 1, -1, 1, -1}};
    constexpr int vy[2][19] = {{0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 1, -1, 1, -1, 0, 0, 0, 0},
                               {0, 0, 0, 1, -1, 1, -1, -1, 1}};
    constexpr int vz[19] = {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, 1, -1};
    int cx = 0, cy = 0, cz = 0;
#pragma unroll
    for (int k = 0; k < NQ; ++k)
        if (i == k) {
            cx = vx[D2][k];
            cy = vy[D2][k];
            cz = D2 ? 0 : vz[k];
        }
    double s = 0.0;
    if (i < NQ) {
        const int q = layout == kAAOdd && i ? ((i & 1) ? i + 1 : i - 1) : i;
        const int from = sum_of_mean(P, u, layout == kAAEven ? 0 : (D2 ? cy : cz));
        const double *p = part + ((int64_t)q * P.nsum + from) * chunks;
#pragma unroll 8
        for (int c = 0; c < chunks; ++c) s += p[c];
    }
    // 0 * infinity is NaN, as in a sum over the sites
    double t[4] = {s, cx * s, cy * s, cz * s};
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
        for (int a = 0; a < 4; ++a) t[a] += __shfl_xor_sync(0xffffffffu, t[a], off);
    }
    // lane a writes value a (FP64 divisions are slow: one per lane)
    const double v = (i == 0 ? t[0] : (i == 1 ? t[1] : (i == 2 ? t[2] : t[3]))) / (double)M;
    if (i == 0) out[u] = rho0 + v;
    else if (i < 4) out[P.n + 3 * u + i - 1] = v;
}

}  // namespace profile

// Chunks per unit: enough blocks to fill the GPU (about eight per SM of 152) as
// long as a block has at least 4096 elements.
inline int profile_chunks(int64_t M, int units, int nq)
{
    const int64_t slots = (int64_t)units * nq, want = (1216 + slots - 1) / slots, most = M / 4096;
    return (int)(want < most ? want : (most < 1 ? 1 : most));
}

// The means of the units of one pass over a box (d2: D2Q9): part is scratch of nq
// nsum chunks doubles, out receives 4 n doubles.  Units of fewer than 2048 elements
// are summed by one warp each (D2Q9 FP32 1500 x 1200: 48 us per call, 58 with blocks),
// but from 1024 on by blocks where there are too few units to fill the SMs with warps
// (48 x 40 x 36: 24.2 us, 26.2 with warps).
template <class S>
cudaError_t launch_profile(const S *buf, int64_t plane, int layout, int64_t M, int units, const profile::Pass &P, bool d2,
                           double rho0, double *part, double *out, cudaStream_t st)
{
    const int nq = d2 ? 9 : Q, chunks = profile_chunks(M, units, nq);
    const int64_t items = (int64_t)P.nsum * nq * chunks;
    constexpr int T = profile::kThreads;
    if (M < 1024 || (M < 2048 && items > 1216))
        profile::k_unit_sums<S, 32><<<(unsigned)((items + T / 32 - 1) / (T / 32)), T, 0, st>>>(buf, plane, M, units, P,
                                                                                               items, chunks, part);
    else
        profile::k_unit_sums<S, T><<<(unsigned)items, T, 0, st>>>(buf, plane, M, units, P, items, chunks, part);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int blocks = (P.n + 3) / 4;
    if (d2) profile::k_unit_means<true><<<blocks, 128, 0, st>>>(part, layout, M, P, chunks, rho0, out);
    else profile::k_unit_means<false><<<blocks, 128, 0, st>>>(part, layout, M, P, chunks, rho0, out);
    return cudaGetLastError();
}

}  // namespace flb
