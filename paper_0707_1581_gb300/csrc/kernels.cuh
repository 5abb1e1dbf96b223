// kernels.cuh -- the stream-collide kernels of the fluctuating D3Q19 library
// (single box and batched), templated on the storage format S; the kernels
// outside the time step are in diag_kernels.cuh.  The step_<format>_<layout>.cu
// files instantiate them; the host runtime calls the launch_* wrappers declared
// in internal.h.
#pragma once

#include "d3q19.cuh"
#include "internal.h"

namespace flb {

// --------------------------------------------------------------------------
// Stream-collide.
// One thread updates V x-consecutive sites of one row (y, z) of one box.
//   AB      pull n_i(r) from slot i at r - c_i of src, store n*_i(r) in slot i at r of dst.
//   AA even read slot i at r, store n*_i(r) in slot opposite(i) at r (in place).
//   AA odd  read slot opposite(i) at r - c_i, store n*_i(r) in slot i at r + c_i (in place).
// In the AA steps every thread writes exactly the locations it read, so the
// in-place update has no races whatever the launch shape.
// --------------------------------------------------------------------------
// n / d for 0 <= n < 2^31 and d >= 1 without a division: with 2^s >= d > 2^(s -
// 1) and m = floor(2^(31 + s) / d) + 1 (which fits 32 bits), m d exceeds 2^(31 +
// s) by at most d <= 2^s, so floor(n m / 2^(31 + s)) is the quotient.
struct FastDiv {
    uint32_t mul;
    int shift;
    FastDiv() = default;
    __host__ explicit FastDiv(int d)
    {
        int s = 0;
        while ((1ll << s) < d) ++s;
        shift = 31 + s;
        mul = (uint32_t)((1ull << shift) / (uint64_t)d + 1);
    }
    __device__ __forceinline__ int quot(int n) const { return (int)(((uint64_t)(uint32_t)n * mul) >> shift); }
};

template <class S>
struct BoxStep {
    const S *src;
    S *dst;
    int nx, ny, nz;
    int warprow;               // batched launch: nx / V divides 32, rows tile the warps (kWarpRow)
    int64_t plane;             // elements between population planes
    uint32_t replica;
    int block0;                // first block of this box in a batched launch
    int z0, nzl;               // single-box launch: planes z0 .. z0 + nzl - 1 (grid.z = nzl)
    int groups, rows;          // threads (of V sites) per row; whole rows per block (kRows)
    FastDiv by_groups, by_ny;  // division by groups and by ny
    CollideConsts<typename Storage<S>::R> K;
    const typename Storage<S>::R *fx;   // the body force F_x(z) of every plane (kernels with a force)
    FLB_VIOL_FIELD
};

// The body force of plane z, from the table that was filled when the context was
// made; FP32 boxes, bound by memory, compute it (about 25 instructions per
// thread).  512 x 512 x 256 FP16 AA odd step 1.100 -> 1.050 ms, 64^3 FP64 101.7 ->
// 96.1 us; 250 x 187 x 93 FP32 100.3 us computed, 101.4 from the table.
template <class S>
__device__ __forceinline__ typename Storage<S>::R force_at(const BoxStep<S> &B, int z)
{
    using R = typename Storage<S>::R;
    if constexpr (sizeof(S) == 4) return B.K.force_amp * sin_pi(B.K.force_phase * R(z));
    else return __ldg(B.fx + z);
}

// When a step's blocks let the next step's blocks start (see d3q19.cuh).  Four
// sites per thread, the launches of many waves: at their own start, so that the
// next step fills the SMs that the last wave leaves.  Fewer sites per thread,
// the boxes of a wave or less: once their loads are back -- any sooner and the
// next step's blocks crowd onto the SMs that happen to be free, which unbalances
// every later step.  FP64, whose collision keeps the SM's FP64 unit busy for
// microseconds: before the stores.  Measured per step, plain launches, at the
// start / after the loads / before the stores (8.20, 6.16, 4.11 and 10.3 us for
// unchained launches): 64^3 FP32 6.26 / 6.02 / 5.94 us, 48^3 FP32 5.32 / 3.80 /
// 4.03, 16^3 FP32 2.26 / 1.69 / 1.92, 16^3 FP64 8.26 / 8.06 / 7.84, 32^3 FP64
// 39.9 / 16.6 / 16.1; V = 4: 96^3 FP32 28.8 / 29.8 / 29.1.
template <class S, int V>
constexpr StartPoint kStart = sizeof(S) == 8 ? kBeforeStores : (V >= 4 ? kAtStart : kAfterLoads);

template <class S, int LAYOUT, int NOISE, bool FORCE, int V>
__device__ __forceinline__ void update_sites(const BoxStep<S> &B, int x0, int y, int z, uint32_t step)
{
    using R = typename Storage<S>::R;
    const int nx = B.nx, ny = B.ny, nz = B.nz;
    const int ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
    const int zm = z == 0 ? nz - 1 : z - 1, zp = z == nz - 1 ? 0 : z + 1;
    // row offsets (in sites) of the nine (y', z') rows the stencil touches
    auto row = [&](int yy, int zz) { return (zz * ny + yy) * nx; };
    auto ysel = [&](int c) { return c > 0 ? ym : (c < 0 ? yp : y); };   // y - c
    auto zsel = [&](int c) { return c > 0 ? zm : (c < 0 ? zp : z); };   // z - c
    auto ysel_push = [&](int c) { return c > 0 ? yp : (c < 0 ? ym : y); };  // y + c
    auto zsel_push = [&](int c) { return c > 0 ? zp : (c < 0 ? zm : z); };
    const uint32_t site_row = (uint32_t)row(y, z);
    static_assert(V == 1, "the scalar path takes one site per thread");
    {
        const int x = x0;
        R g[16];
        if (NOISE) draw_normals<R>(B.K, site_row + (uint32_t)x, step, B.replica, g);
        wait_for_previous_step();
        const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
        auto xsel = [&](int c) { return c > 0 ? xm : (c < 0 ? xp : x); };
        auto xsel_push = [&](int c) { return c > 0 ? xp : (c < 0 ? xm : x); };
        R f[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            int idx, slot;
            if (LAYOUT == kAAEven) {
                idx = (int)site_row + x;
                slot = i;
            } else {
                idx = row(ysel(vel_y(i)), zsel(vel_z(i))) + xsel(vel_x(i));
                slot = LAYOUT == kAB ? i : opposite(i);
            }
            const S *p = B.src + (int64_t)slot * B.plane + idx;
            f[i] = Storage<S>::load(load_ro(FLB_GUARD_LD(B, p, 1)));
        }
        if constexpr (kStart<S, V> == kAfterLoads) let_next_step_start();
        const R Fx = FORCE ? force_at(B, z) : R(0);
        if constexpr (sizeof(R) == 8) collide64<NOISE, FORCE, true>(f, B.K, site_row + (uint32_t)x, step, B.replica, Fx, g);
        else collide<R, NOISE, FORCE, true>(f, B.K, site_row + (uint32_t)x, step, B.replica, Fx, g);
        stochastic_round<S>(f, site_row + (uint32_t)x, step, B.replica, B.K.rk0, B.K.rk1);
        if constexpr (kStart<S, V> == kBeforeStores) let_next_step_start();
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            int idx, slot;
            if (LAYOUT == kAB) {
                idx = (int)site_row + x;
                slot = i;
            } else if (LAYOUT == kAAEven) {
                idx = (int)site_row + x;
                slot = opposite(i);
            } else {
                idx = row(ysel_push(vel_y(i)), zsel_push(vel_z(i))) + xsel_push(vel_x(i));
                slot = i;
            }
            S *p = B.dst + (int64_t)slot * B.plane + idx;
            if (FLB_GUARD_ST(B, p, 1)) *p = Storage<S>::store(f[i]);
        }
    }
}

// --------------------------------------------------------------------------
// Vectorised update: one thread owns V x-consecutive sites x0..x0+V-1 of row
// (y, z) (nx % V == 0, x0 % V == 0), so every population plane is read and
// written with one aligned V-wide access.  A shift of the source (pull) or
// destination (AA odd push) by c_x = +-1 is resolved with a warp shuffle of the
// neighbouring thread's edge element; only threads at a row end or a warp or
// block-row edge fall back to one scalar access for that element.  All 32
// lanes of a warp reach every shuffle (inactive lanes work on a clamped,
// in-bounds position and skip their stores).
// --------------------------------------------------------------------------
template <int BYTES>
struct RawVec;
template <>
struct RawVec<4> {
    using T = uint32_t;
};
template <>
struct RawVec<8> {
    using T = uint2;
};
template <>
struct RawVec<16> {
    using T = uint4;
};

template <class S, int V>
__device__ __forceinline__ void load_vec(const S *p, S (&out)[V])
{
    using T = typename RawVec<sizeof(S) * V>::T;
    const T raw = *reinterpret_cast<const T *>(p);
    const S *e = reinterpret_cast<const S *>(&raw);
#pragma unroll
    for (int v = 0; v < V; ++v) out[v] = e[v];
}

template <class S, int V>
__device__ __forceinline__ void store_vec(S *p, const S (&in)[V])
{
    using T = typename RawVec<sizeof(S) * V>::T;
    T raw;
    S *e = reinterpret_cast<S *>(&raw);
#pragma unroll
    for (int v = 0; v < V; ++v) e[v] = in[v];
    *reinterpret_cast<T *>(p) = raw;
}

// Stores guarded by a predicate without a branch, so that the edge lanes of
// a warp do not split it (hand-written PTX: one predicated st.global).
__device__ __forceinline__ void st_if(bool p, void *a, uint16_t v)
{
    asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %0, 0;\n @q st.global.b16 [%1], %2;\n}" ::"r"((int)p), "l"(a),
                 "h"(v)
                 : "memory");
}
__device__ __forceinline__ void st_if(bool p, void *a, uint32_t v)
{
    asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %0, 0;\n @q st.global.b32 [%1], %2;\n}" ::"r"((int)p), "l"(a),
                 "r"(v)
                 : "memory");
}
__device__ __forceinline__ void st_if(bool p, void *a, uint64_t v)
{
    asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %0, 0;\n @q st.global.b64 [%1], %2;\n}" ::"r"((int)p), "l"(a),
                 "l"(v)
                 : "memory");
}
__device__ __forceinline__ void st_if(bool p, void *a, uint2 v)
{
    asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %0, 0;\n @q st.global.v2.b32 [%1], {%2, %3};\n}" ::"r"((int)p),
                 "l"(a), "r"(v.x), "r"(v.y)
                 : "memory");
}
__device__ __forceinline__ void st_if(bool p, void *a, uint4 v)
{
    asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %0, 0;\n @q st.global.v4.b32 [%1], {%2, %3, %4, %5};\n}" ::"r"((int)p),
                 "l"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
}

template <int BYTES>
struct RawScalar;
template <>
struct RawScalar<2> {
    using T = uint16_t;
};
template <>
struct RawScalar<4> {
    using T = uint32_t;
};
template <>
struct RawScalar<8> {
    using T = uint64_t;
};

// One element if p.
template <class S>
__device__ __forceinline__ void store_one_if(bool p, S *a, S v)
{
    using T = typename RawScalar<sizeof(S)>::T;
    st_if(p, a, *reinterpret_cast<const T *>(&v));
}

// V elements (aligned) if p.
template <class S, int V>
__device__ __forceinline__ void store_vec_if(bool p, S *a, const S (&in)[V])
{
    using T = typename RawVec<sizeof(S) * V>::T;
    T raw;
    S *e = reinterpret_cast<S *>(&raw);
#pragma unroll
    for (int v = 0; v < V; ++v) e[v] = in[v];
    st_if(p, a, raw);
}

// V elements (aligned) if p, as an ordinary store: for the whole-vector stores
// the compiler can fold the address arithmetic into the store's addressing.
template <class S, int V>
__device__ __forceinline__ void store_vec_when(bool p, S *a, const S (&in)[V])
{
    if (p) store_vec<S, V>(a, in);
}

template <class R>
__device__ __forceinline__ R shfl_up1(R v)
{
    return __shfl_up_sync(0xffffffffu, v, 1);
}
template <class R>
__device__ __forceinline__ R shfl_down1(R v)
{
    return __shfl_down_sync(0xffffffffu, v, 1);
}

// How update_vec gets the elements that cross from one thread's V sites into
// the next's (the x-shift by c_x = +-1).
//   kEdges    lane - 1 and lane + 1 by shuffle where they own the adjacent
//             sites, else by scalar accesses; any shape.
//   kEdgeRow  the same, in blocks that lie in one row.
//   kOneRow   the block is one box row of whole warps: shuffles inside a warp,
//             a shared-memory exchange across warps and around the periodic row
//             end; every lane reads and writes only whole aligned vectors.
//   kRagRow   the block is one box row that is not whole warps: as kOneRow, with
//             an exchange slot for the row end besides the one per warp end.
//   kRows     the block is several whole box rows: as kRagRow, a slot per row.
//   kWarpRow  a row is g = nx / V consecutive lanes and g divides 32, so rows
//             tile the warps: every neighbour element comes by an indexed
//             shuffle, with no edge access and no shared memory.
// FP32, bound by memory, gains most from the whole vectors: 250 x 187 x 93 AA
// 117 us per step with kEdges, 100 with kRagRow; 300 x 200 x 60 AB 96 / 84 (kRows);
// 640 x 320 x 40 AB 207 / 181 (kOneRow).  The 16-bit formats, bound by
// instructions, only where no lane idles: 300 x 200 x 60 AB 61.7 / 66.3, 400 x
// 100 x 100 64.5 / 76.1 (kRagRow, 100 of 128 lanes), 640 wide 132 / 129; two sites
// per thread 87 / 77 (250 wide AA).  FP64 likewise: 90 x 100 x 110 368 / 397 (90 of
// 96 lanes), 72^3 154 / 145.  (set_exchange in launch_shape.h decides.)
enum Exchange : int { kEdges = 0, kOneRow = 1, kRows = 2, kWarpRow = 3, kRagRow = 4, kEdgeRow = 5 };

// The block's exchange memory: what a warp (kOneRow) or a warp or row (kRows)
// hands over its ends, in the load phase (l*, as stored) and in the store phase
// (s*).
constexpr int kXchWarps = 8;       // warps per block, at most (rows: kXchRows)
template <class S, int XCH>
struct RowExchange {
    using R = typename Storage<S>::R;
    static constexpr int kRowSlots = XCH == kRows ? kXchRows : 1;
    static constexpr int kSlots = XCH == kOneRow ? kXchWarps : kRowSlots + kXchWarps;
    S l_last[Q][kSlots];    // last element of the vector (pull from x - 1)
    S l_first[Q][kSlots];   // first element (pull from x + 1)
    R s_last[Q][kSlots];    // value pushed to x + 1 across the end
    R s_first[Q][kSlots];   // value pushed to x - 1 across the end
};

// A thread's place in its block's rows (kOneRow, kRows): which ends it owns,
// and the exchange slots that it writes (mine_*) and reads (from_*).  A row end
// has the row's slot; a warp end inside a row has the warp's.  A thread beyond the
// block's rows gets slots inside the arrays too; what it reads there is not used.
struct RowPlace {
    bool give_last, give_first;    // the right (left) neighbour cannot reach this thread by shuffle
    bool take_left, take_right;    // the left (right) neighbour's element comes from the exchange
    int mine_last, mine_first, from_left, from_right;
};
template <int XCH>
__host__ __device__ __forceinline__ RowPlace row_place(int lane, int warp, int nwarp, int tx, int g, int row)
{
    RowPlace p;
    if constexpr (XCH == kOneRow) {
        p.give_last = p.take_right = lane == 31;
        p.give_first = p.take_left = lane == 0;
        p.mine_last = p.mine_first = warp;
        p.from_left = warp == 0 ? nwarp - 1 : warp - 1;
        p.from_right = warp == nwarp - 1 ? 0 : warp + 1;
    } else {
        constexpr int kRowSlots = XCH == kRows ? kXchRows : 1;
        const bool start = tx == 0, end = tx == g - 1;
        p.give_last = p.take_right = lane == 31 || end;
        p.give_first = p.take_left = lane == 0 || start;
        p.mine_last = end ? row : kRowSlots + warp;
        p.mine_first = start ? row : kRowSlots + warp;
        p.from_left = start ? row : kRowSlots + (lane == 0 ? warp - 1 : warp);
        const int next = warp + 1 < kXchWarps ? warp + 1 : warp;   // the last warp's last lane ends a row, or is idle
        p.from_right = end ? row : kRowSlots + (lane == 31 ? next : warp);
    }
    return p;
}

// OFF32: every element offset of the box's buffer (Q planes) fits in 32 bits,
// so an address is one 32-bit offset (slot, row and x together) added to the
// buffer pointer, instead of 64-bit arithmetic per access.
// row: the thread's row within its block (kRows).
template <class S, int LAYOUT, int NOISE, bool FORCE, int V, int XCH = kEdges, bool OFF32 = false>
__device__ __forceinline__ void update_vec(const BoxStep<S> &B, int x0, int y, int z, bool active, bool left_in_warp,
                                           bool right_in_warp, uint32_t step, RowExchange<S, XCH> *xch = nullptr,
                                           int row = 0)
{
    constexpr bool FULLROW = XCH == kOneRow || XCH == kRows || XCH == kRagRow, WARPROW = XCH == kWarpRow;
    using R = typename Storage<S>::R;
    // element (slot, row offset + x) of the source / destination buffer
    auto src_at = [&](int slot, int off) -> const S * {
        if constexpr (OFF32) return B.src + ((uint32_t)slot * (uint32_t)B.plane + (uint32_t)off);
        else return B.src + (int64_t)slot * B.plane + off;
    };
    auto dst_at = [&](int slot, int off) -> S * {
        if constexpr (OFF32) return B.dst + ((uint32_t)slot * (uint32_t)B.plane + (uint32_t)off);
        else return B.dst + (int64_t)slot * B.plane + off;
    };
    const int nx = B.nx, ny = B.ny, nz = B.nz;
    // row offsets: yo[1 + d] = ((y + d) mod ny) nx, zo[1 + d] = ((z + d) mod nz) nx ny
    const int yo[3] = {(y == 0 ? ny - 1 : y - 1) * nx, y * nx, (y == ny - 1 ? 0 : y + 1) * nx};
    const int nxy = nx * ny;
    const int zo[3] = {(z == 0 ? nz - 1 : z - 1) * nxy, z * nxy, (z == nz - 1 ? 0 : z + 1) * nxy};
    const uint32_t site0 = (uint32_t)(zo[1] + yo[1]) + (uint32_t)x0;
    // Two sites per thread in rows of whole warps (the small boxes): the normals,
    // which need no stored state, before the wait; four sites' would not fit
    // beside the populations, and a step of many waves runs 5 % slower with the
    // loads behind them (250 x 187 x 93 FP32, 131 against 125 us).
    constexpr bool kPaired = sizeof(R) == 4 && sizeof(S) == 2 && V % 2 == 0;
    constexpr bool kDrawn = NOISE && V == 2 && WARPROW;
    using G = typename std::conditional<kPaired, F2, R>::type;
    constexpr int NG = kPaired ? V / 2 : V;
    G g[kDrawn ? NG : 1][16];
    if constexpr (kDrawn && kPaired) {
        draw_normals<F2>(B.K, make_uint2(site0, site0 + 1), step, B.replica, g[0]);
    } else if constexpr (kDrawn) {
#pragma unroll
        for (int v = 0; v < V; ++v) draw_normals<R>(B.K, site0 + v, step, B.replica, g[v]);
    }
    wait_for_previous_step();

    // a neighbour's element comes by shuffle only inside the same row
    const bool shl = left_in_warp && x0 != 0;          // lane - 1 owns x0 - V .. x0 - 1
    const bool shr = right_in_warp && x0 + V != nx;    // lane + 1 owns x0 + V .. x0 + 2V - 1
    const int x_left = x0 == 0 ? nx - 1 : x0 - 1;      // element left of the group (periodic)
    const int x_right = x0 + V == nx ? 0 : x0 + V;     // element right of the group (periodic)
    // every lane reads its edge element with the vector (no wait behind the
    // shuffle, no divergence); lanes that get it by shuffle re-read a word of
    // their own vector instead
    const int x_lload = shl ? x0 : x_left;
    const int x_rload = shr ? x0 + V - 1 : x_right;

    // 1. issue every load of the 19 planes (vector + edge element) before
    //    any shuffle, so that all of them are in flight together
    S raw[Q][V];
    S edge[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const int cx = vel_x(i), cy = vel_y(i), cz = vel_z(i);
        int ro, slot;
        if (LAYOUT == kAAEven) {
            ro = zo[1] + yo[1];
            slot = i;
        } else {
            ro = zo[1 - cz] + yo[1 - cy];   // pull from r - c_i
            slot = LAYOUT == kAB ? i : opposite(i);
        }
        load_vec<S, V>(FLB_GUARD_LD(B, src_at(slot, ro + x0), V), raw[i]);
        if (!FULLROW && !WARPROW && LAYOUT != kAAEven && cx > 0) edge[i] = load_ro(FLB_GUARD_LD(B, src_at(slot, ro + x_lload), 1));
        if (!FULLROW && !WARPROW && LAYOUT != kAAEven && cx < 0) edge[i] = load_ro(FLB_GUARD_LD(B, src_at(slot, ro + x_rload), 1));
    }
    const int lane = (threadIdx.y * blockDim.x + threadIdx.x) & 31;   // 2-D blocks: kWarpRow only
    // WARPROW source lanes of the left (x - 1) and right (x + 1) neighbour, periodic in the row
    const int gl = nx / V;
    const int lane_l = WARPROW ? (x0 != 0 ? lane - 1 : lane + gl - 1) : 0;
    const int lane_r = WARPROW ? (x0 + V != nx ? lane + 1 : lane - gl + 1) : 0;
    const RowPlace at = FULLROW ? row_place<XCH>(lane, (int)threadIdx.x >> 5, (int)blockDim.x >> 5, x0 / V, gl, row)
                                : RowPlace{};
    if constexpr (FULLROW && LAYOUT != kAAEven) {
        // publish the end elements, then read the neighbours' (periodic in the row)
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            if (vel_x(i) > 0 && at.give_last && (XCH == kOneRow || active)) xch->l_last[i][at.mine_last] = raw[i][V - 1];
            if (vel_x(i) < 0 && at.give_first && (XCH == kOneRow || active)) xch->l_first[i][at.mine_first] = raw[i][0];
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            if (vel_x(i) > 0) edge[i] = xch->l_last[i][at.from_left];
            if (vel_x(i) < 0) edge[i] = xch->l_first[i][at.from_right];
        }
    }
    // 2. shift the planes with c_x != 0 by one site
    const bool use_left = FULLROW ? !at.take_left : shl;
    const bool use_right = FULLROW ? !at.take_right : shr;
    R f[V][Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const int cx = vel_x(i);
        if (LAYOUT == kAAEven || cx == 0) {
#pragma unroll
            for (int v = 0; v < V; ++v) f[v][i] = Storage<S>::load(raw[i][v]);
        } else if (cx > 0) {   // pull from x - 1
            if constexpr (WARPROW) {
                f[0][i] = __shfl_sync(0xffffffffu, Storage<S>::load(raw[i][V - 1]), lane_l);
            } else {
                const R via = shfl_up1(Storage<S>::load(raw[i][V - 1]));
                f[0][i] = use_left ? via : Storage<S>::load(edge[i]);
            }
#pragma unroll
            for (int v = 1; v < V; ++v) f[v][i] = Storage<S>::load(raw[i][v - 1]);
        } else {               // pull from x + 1
#pragma unroll
            for (int v = 0; v < V - 1; ++v) f[v][i] = Storage<S>::load(raw[i][v + 1]);
            if constexpr (WARPROW) {
                f[V - 1][i] = __shfl_sync(0xffffffffu, Storage<S>::load(raw[i][0]), lane_r);
            } else {
                const R via = shfl_down1(Storage<S>::load(raw[i][0]));
                f[V - 1][i] = use_right ? via : Storage<S>::load(edge[i]);
            }
        }
    }

    if constexpr (kStart<S, V> == kAfterLoads) let_next_step_start();
    const R Fx = FORCE ? force_at(B, z) : R(0);
    // 16-bit formats (issue-bound): two sites per collision in the paired FP32
    // instructions; FP32 storage is bound by HBM and keeps the one-site form,
    // whose odd AA step measured faster
    if constexpr (kPaired) {
#pragma unroll
        for (int v = 0; v < V; v += 2) {
            F2 p[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i) p[i] = F2(f[v][i], f[v + 1][i]);
            collide<F2, NOISE, FORCE, kDrawn>(p, B.K, make_uint2(site0 + v, site0 + v + 1), step, B.replica, F2(Fx),
                                              g[kDrawn ? v / 2 : 0]);
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                f[v][i] = p[i].v.x;
                f[v + 1][i] = p[i].v.y;
            }
        }
    } else {
#pragma unroll
        for (int v = 0; v < V; ++v) {
            if constexpr (sizeof(R) == 8)
                collide64<NOISE, FORCE, kDrawn>(f[v], B.K, site0 + v, step, B.replica, Fx, g[kDrawn ? v : 0]);
            else
                collide<R, NOISE, FORCE, kDrawn>(f[v], B.K, site0 + v, step, B.replica, Fx, g[kDrawn ? v : 0]);
        }
    }
#pragma unroll
    for (int v = 0; v < V; ++v) stochastic_round<S>(f[v], site0 + v, step, B.replica, B.K.rk0, B.K.rk1);

    if constexpr (kStart<S, V> == kBeforeStores) let_next_step_start();
    R pushed[Q];   // FULLROW, AA odd: the value that crosses into this thread's vector through the exchange
    if constexpr (FULLROW && LAYOUT == kAAOdd) {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            if (vel_x(i) > 0 && at.give_last && (XCH == kOneRow || active)) xch->s_last[i][at.mine_last] = f[V - 1][i];
            if (vel_x(i) < 0 && at.give_first && (XCH == kOneRow || active)) xch->s_first[i][at.mine_first] = f[0][i];
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            pushed[i] = R(0);
            if (vel_x(i) > 0) pushed[i] = xch->s_last[i][at.from_left];
            if (vel_x(i) < 0) pushed[i] = xch->s_first[i][at.from_right];
        }
    }
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const int cx = vel_x(i), cy = vel_y(i), cz = vel_z(i);
        if (WARPROW && LAYOUT == kAAOdd && cx != 0) {
            // whole aligned vectors: the element crossing a lane edge comes from the neighbour lane
            S *base = B.dst + (int64_t)i * B.plane + zo[1 + cz] + yo[1 + cy];
            S out[V];
            if (cx > 0) {   // site x goes to x + 1
                out[0] = Storage<S>::store(__shfl_sync(0xffffffffu, f[V - 1][i], lane_l));
#pragma unroll
                for (int v = 1; v < V; ++v) out[v] = Storage<S>::store(f[v - 1][i]);
            } else {        // site x goes to x - 1
#pragma unroll
                for (int v = 0; v < V - 1; ++v) out[v] = Storage<S>::store(f[v + 1][i]);
                out[V - 1] = Storage<S>::store(__shfl_sync(0xffffffffu, f[0][i], lane_r));
            }
            store_vec_when<S, V>(active && FLB_GUARD_ST(B, base + x0, V), base + x0, out);
            continue;
        }
        if (FULLROW && LAYOUT == kAAOdd && cx != 0) {
            // whole aligned vectors only: the element that crosses the warp edge came through the exchange
            S out[V];
            if (cx > 0) {   // site x goes to x + 1
                const R from_left = shfl_up1(f[V - 1][i]);
                out[0] = Storage<S>::store(at.take_left ? pushed[i] : from_left);
#pragma unroll
                for (int v = 1; v < V; ++v) out[v] = Storage<S>::store(f[v - 1][i]);
            } else {        // site x goes to x - 1
                const R from_right = shfl_down1(f[0][i]);
#pragma unroll
                for (int v = 0; v < V - 1; ++v) out[v] = Storage<S>::store(f[v + 1][i]);
                out[V - 1] = Storage<S>::store(at.take_right ? pushed[i] : from_right);
            }
            S *p = dst_at(i, zo[1 + cz] + yo[1 + cy] + x0);
            store_vec_when<S, V>(active && FLB_GUARD_ST(B, p, V), p, out);
            continue;
        }
        if (LAYOUT != kAAOdd) {
            // AB: slot i at r;  AA even: slot opposite(i) at r
            S *p = dst_at(LAYOUT == kAB ? i : opposite(i), zo[1] + yo[1] + x0);
            S out[V];
#pragma unroll
            for (int v = 0; v < V; ++v) out[v] = Storage<S>::store(f[v][i]);
            store_vec_when<S, V>(active && FLB_GUARD_ST(B, p, V), p, out);
        } else {
            // AA odd: push population i to slot i at r + c_i
            S *base = B.dst + (int64_t)i * B.plane + zo[1 + cz] + yo[1 + cy];
            if (cx == 0) {
                S out[V];
#pragma unroll
                for (int v = 0; v < V; ++v) out[v] = Storage<S>::store(f[v][i]);
                store_vec_if<S, V>(active && FLB_GUARD_ST(B, base + x0, V), base + x0, out);
            } else if (cx > 0) {   // site x goes to x + 1
                const R from_left = shfl_up1(f[V - 1][i]);
                S out[V];
                out[0] = Storage<S>::store(from_left);
#pragma unroll
                for (int v = 1; v < V; ++v) out[v] = Storage<S>::store(f[v - 1][i]);
                store_vec_if<S, V>(active && shl && FLB_GUARD_ST(B, base + x0, V), base + x0, out);
                // without the left neighbour: elements x0+1 .. x0+V-1 one by one
#pragma unroll
                for (int v = 1; v < V; ++v) store_one_if<S>(active && !shl && FLB_GUARD_ST(B, base + x0 + v, 1), base + x0 + v, out[v]);
                store_one_if<S>(active && !shr && FLB_GUARD_ST(B, base + x_right, 1), base + x_right, Storage<S>::store(f[V - 1][i]));
            } else {               // site x goes to x - 1
                const R from_right = shfl_down1(f[0][i]);
                S out[V];
#pragma unroll
                for (int v = 0; v < V - 1; ++v) out[v] = Storage<S>::store(f[v + 1][i]);
                out[V - 1] = Storage<S>::store(from_right);
                store_vec_if<S, V>(active && shr && FLB_GUARD_ST(B, base + x0, V), base + x0, out);
#pragma unroll
                for (int v = 0; v < V - 1; ++v) store_one_if<S>(active && !shr && FLB_GUARD_ST(B, base + x0 + v, 1), base + x0 + v, out[v]);
                store_one_if<S>(active && !shl && FLB_GUARD_ST(B, base + x_left, 1), base + x_left, Storage<S>::store(f[0][i]));
            }
        }
    }
}

__device__ __forceinline__ uint32_t step_of(const uint32_t *step_ptr, uint32_t step)
{
    return step_ptr ? __ldg(step_ptr) + step : step;
}

// Block b of a kRows launch: rows b B.rows .. of the box's planes z0 .. z0 + nzl - 1,
// thread tid on group tid mod B.groups of row tid / B.groups.
template <class S, int LAYOUT, int NOISE, bool FORCE, int V, bool OFF32>
__device__ __forceinline__ void update_rows(const BoxStep<S> &B, int tid, int b, uint32_t step,
                                            RowExchange<S, kRows> &xch)
{
    const int tr = B.by_groups.quot(tid), tx = tid - tr * B.groups;
    const int first = b * B.rows, nrows = B.ny * B.nzl;
    const bool active = tr < B.rows && first + tr < nrows;
    const int row = active ? first + tr : min(first, nrows - 1);   // in bounds for every lane
    const int zr = B.by_ny.quot(row);
    update_vec<S, LAYOUT, NOISE, FORCE, V, kRows, OFF32>(B, V * tx, row - zr * B.ny, B.z0 + zr, active, true, true, step,
                                                         &xch, min(tr, kXchRows - 1));
}

// One box; a thread updates the V sites x0 .. x0 + V - 1 of row (y, z); V > 1
// needs nx % V == 0 and blocks of whole warps.
//   kEdges   (and V = 1) a 1-D grid over the groups of V sites of all the rows
//            of the launch, so that no lane idles at a row end.
//   kRows    a 1-D grid over the rows of the launch (y + ny z), B.rows whole
//            rows of B.groups threads per block; the threads beyond them (less
//            than a warp, or rows past the last) only keep the warps whole.
//   the rest grid (x, y, z), block (bx, by); kOneRow, kRagRow, kEdgeRow: y =
//            blockIdx.y, so the row offsets of the nine neighbour rows are the
//            same for the whole block (1000 x 100 x 40 FP16 AB: 65.6 us per step
//            with kEdgeRow, 71.6 with kEdges).
template <class S, int LAYOUT, int NOISE, bool FORCE, int V, int XCH, bool OFF32>
__device__ __forceinline__ void stream_collide_box(const BoxStep<S> &B, const uint32_t *step_ptr, uint32_t step)
{
    if constexpr (kStart<S, V> == kAtStart) let_next_step_start();
    const int tid = (int)threadIdx.x, lane = tid & 31;
    if constexpr (XCH == kRows) {
        __shared__ RowExchange<S, XCH> xch;
        update_rows<S, LAYOUT, NOISE, FORCE, V, OFF32>(B, tid, (int)blockIdx.x, step_of(step_ptr, step), xch);
    } else if constexpr (XCH == kEdges) {
        const uint32_t items = (uint32_t)B.groups * (uint32_t)(B.ny * B.nzl);
        const uint32_t it = blockIdx.x * blockDim.x + threadIdx.x;
        const bool active = it < items;
        const int item = (int)(active ? it : items - 1);   // idle lanes work on the last group, store nothing
        const int row = B.by_groups.quot(item), xg = item - row * B.groups;
        const int zr = B.by_ny.quot(row);
        if constexpr (V == 1) {
            if (active)
                update_sites<S, LAYOUT, NOISE, FORCE, 1>(B, xg, row - zr * B.ny, B.z0 + zr, step_of(step_ptr, step));
        } else {
            // consecutive lanes own consecutive groups: lane - 1 holds x0 - V whenever x0 > 0
            update_vec<S, LAYOUT, NOISE, FORCE, V, XCH, OFF32>(B, V * xg, row - zr * B.ny, B.z0 + zr, active, lane > 0,
                                                               lane < 31, step_of(step_ptr, step));
        }
    } else if constexpr (XCH == kWarpRow) {
        const int y = (int)(blockIdx.y * blockDim.y + threadIdx.y);
        update_vec<S, LAYOUT, NOISE, FORCE, V, XCH, OFF32>(B, V * tid, min(y, B.ny - 1), B.z0 + (int)blockIdx.z, y < B.ny,
                                                           true, true, step_of(step_ptr, step));
    } else if constexpr (XCH == kEdgeRow) {
        const int x0 = V * (int)(blockIdx.x * blockDim.x + threadIdx.x);
        update_vec<S, LAYOUT, NOISE, FORCE, V, XCH, OFF32>(B, min(x0, B.nx - V), (int)blockIdx.y, B.z0 + (int)blockIdx.z,
                                                           x0 < B.nx, lane > 0, lane < 31, step_of(step_ptr, step));
    } else {
        __shared__ RowExchange<S, XCH> xch;
        const bool active = XCH == kOneRow || tid < B.groups;
        update_vec<S, LAYOUT, NOISE, FORCE, V, XCH, OFF32>(B, V * (XCH == kOneRow ? tid : min(tid, B.groups - 1)),
                                                           (int)blockIdx.y, B.z0 + (int)blockIdx.z, active, true, true,
                                                           step_of(step_ptr, step), &xch);
    }
}

// Registers: 512 threads per SM (at most 128 each) with four sites per thread --
// left free, many variants took 130 to 176, which leaves room for three or two
// blocks of 128 threads instead of four (the stochastically rounded AA odd step
// took 130 and ran 15 % slower) -- and 768 (at most 85) with two, which took 120
// (250 x 187 x 93 AA, per step: FP16 90.6 -> 77.3 us, FP32 107 -> 100; 64
// registers: 76.8 and 100.5).  The small boxes of kWarpRow hold their normals
// too and keep what they take (64^3 FP32 AA 6.2 us, 6.8 with 85).
template <class S, int V, int XCH>
constexpr int kMinBlocks = sizeof(S) == 8 ? 1 : (V == 4 ? 2 : (V == 2 && XCH != kWarpRow ? 3 : 1));

template <class S, int LAYOUT, int NOISE, bool FORCE, int V, int XCH = kEdges, bool OFF32 = false>
__global__ void __launch_bounds__(256, kMinBlocks<S, V, XCH>) k_stream_collide(const BoxStep<S> B,
                                                                             const uint32_t *step_ptr, uint32_t step)
{
    stream_collide_box<S, LAYOUT, NOISE, FORCE, V, XCH, OFF32>(B, step_ptr, step);
}

// Many boxes in one 1-D grid: box b owns the blocks from block0 on.  FP32 boxes
// whose rows do not tile the warps but nearly fill the blocks (batch_rows) take whole
// rows per block (kRows: 12 boxes of 96^3, AB, 45.3 GLUPS against 41.0 with the scalar
// accesses of kEdges); in the other boxes the threads are packed densely: thread item k = (block - block0) T
// + tid owns the V sites of x-group k mod groups (nx / V groups per row) of row k
// / groups, so a warp may span several short rows and no lane idles at a row
// end.  The box table is a kernel parameter (constant bank, at most ~31 KB);
// batches larger than one table are split into several launches.
template <class S>
constexpr int batch_chunk()
{
    constexpr int n = (int)(31000 / sizeof(BoxStep<S>));
    return n > 64 ? 64 : n;
}

template <class S>
struct BatchParams {
    int nboxes;
    int pad_;
    BoxStep<S> boxes[batch_chunk<S>()];
};

// Registers of the batch kernel, as blocks of 256 threads that an SM must hold.
// Measured per format with 1 to 5 blocks, us per step (blocks in brackets):
//   V = 2, 24 boxes of 50^3: FP16 AB 69.6 (2) 63.5 (3) 57.3 (4), AA 61.4 (3) 62.0 (4);
//     bfloat16 AB 64.4 / 58.0, AA 62.9 / 62.0; stochastic AB 78.8 / 79.5, AA 82.3 / 83.8;
//     FP32 AB 86.6 (2) 76.5 (3) 70.1 (4), AA 77.2 (3) 79.1 (4)
//   V = 2, 16 boxes of 24^3, less than a wave: FP16 AB 5.90 (3) 6.25 (4), AA 6.04 / 7.05;
//     11 boxes of 32^3, whose rows tile the warps: FP32 AB 8.72 / 10.0, FP16 AA 8.51 / 9.14
//   V = 1, 8 boxes of 65^3, whose threads hold their normals over the wait (82 to 90
//     registers when left free): stochastic AB 76.0 (2) 74.3 (4) 71.2 (5); FP16 AB 61.6 /
//     58.9 / 56.5; FP32 AB 60.7 (3) 54.1 (5); AA 75.5 with 5, 74.5 free (stochastic),
//     86.6 / 59.0 (FP16), where five blocks spill
// So AB steps of two sites take four blocks, but three in launches of a wave or less and
// in FP32 where every box's rows tile the warps (step_batch in step_impl.cuh).
template <class S, int LAYOUT, int V>
constexpr int kBatchMinBlocks = sizeof(S) == 8 ? 1
                                : V == 4       ? kMinBlocks<S, V, kEdges>
                                : V == 1       ? (LAYOUT == kAB ? 5 : 1)
                                : Storage<S>::stochastic || LAYOUT != kAB ? 3 : 4;

template <class S, int LAYOUT, int NOISE, bool FORCE, int V, int MIN_BLOCKS = kBatchMinBlocks<S, LAYOUT, V>>
__global__ void __launch_bounds__(256, MIN_BLOCKS)
k_stream_collide_batch(const __grid_constant__ BatchParams<S> P, const uint32_t *step_ptr, uint32_t step)
{
    if constexpr (kStart<S, V> == kAtStart) let_next_step_start();
    // last box with block0 <= blockIdx.x (the same for the whole block)
    int lo = 0, hi = P.nboxes - 1;
    const int b = (int)blockIdx.x;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (P.boxes[mid].block0 <= b) lo = mid;
        else hi = mid - 1;
    }
    const BoxStep<S> &sb = P.boxes[lo];
    const int tid = (int)threadIdx.x;
    if constexpr (V > 1 && sizeof(S) == 4) {
        __shared__ RowExchange<S, kRows> xch;
        if (sb.rows > 0) {
            update_rows<S, LAYOUT, NOISE, FORCE, V, false>(sb, tid, b - sb.block0, step_of(step_ptr, step), xch);
            return;
        }
    }
    const int total = sb.groups * sb.ny * sb.nz;             // x-groups of the box
    const int item = (b - sb.block0) * (int)blockDim.x + tid;
    const bool active = item < total;
    const int it = active ? item : total - 1;                // idle lanes work on the last group, store nothing
    const int row = sb.by_groups.quot(it), z = sb.by_ny.quot(row);
    const int y = row - z * sb.ny, x0 = V * (it - row * sb.groups);
    if constexpr (V == 1) {
        if (!active) return;
        update_sites<S, LAYOUT, NOISE, FORCE, 1>(sb, x0, y, z, step_of(step_ptr, step));
    } else {
        // consecutive lanes own consecutive x-groups: lane - 1 holds x0 - V whenever x0 > 0
        const int lane = tid & 31;
        if (sb.warprow)
            update_vec<S, LAYOUT, NOISE, FORCE, V, kWarpRow>(sb, x0, y, z, active, lane > 0, lane < 31,
                                                                step_of(step_ptr, step));
        else
            update_vec<S, LAYOUT, NOISE, FORCE, V>(sb, x0, y, z, active, lane > 0, lane < 31, step_of(step_ptr, step));
    }
}

__global__ void k_advance_step(uint32_t *step_ptr, uint32_t by);

}  // namespace flb
