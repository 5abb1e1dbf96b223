// launch_shape.h -- which launch shape a context steps its boxes with: what fits
// them, the automatic choice and the autotuner's candidates.  Host code without
// CUDA calls.
#pragma once

#include <algorithm>
#include <cstdint>
#include <vector>

#include "flb.h"
#include "internal.h"

namespace flb {

// What a launch shape depends on.
struct LaunchBoxes {
    int store;              // flb_store_t
    bool d2;                // D2Q9
    std::vector<int> nx;    // of every box
    int64_t sites;          // of all boxes
};

// Largest usable sites-per-thread <= V: the vector path needs nx % V == 0 in
// every box, at most 16-byte accesses (FP64: V <= 2) and whole warps (its
// neighbour exchange is a full-warp shuffle), i.e. bx * by % 32 == 0.
inline int usable_V(const LaunchBoxes &B, int V, int bx, int by)
{
    if ((bx * by) % 32 != 0) return 1;
    if (B.store == FLB_STORE_F64 && V > 2) V = 2;
    for (;;) {
        bool ok = true;
        for (int nx : B.nx) ok = ok && (nx % V == 0);
        if (ok || V == 1) return V;
        V /= 2;
    }
}

// Which exchange the single-box kernel uses for a launch shape (measured, see
// Exchange in kernels.cuh): rows that tile the warps; as many whole rows as the
// block's threads hold -- FP32 always, the formats bound by instructions (16-bit,
// FP64) where hardly a lane idles --; blocks that lie in one row where they cover
// it with few idle lanes; else threads over the whole box.
inline void set_exchange(const LaunchBoxes &B, Launch &L)
{
    L.warprow = L.edgerow = false;
    L.rows = 0;
    if (B.nx.size() != 1 || L.V < 2 || B.d2) return;
    const int V = (B.store == FLB_STORE_F64 && L.V == 4) ? 2 : L.V;
    const int nx = B.nx[0], T = L.bx * L.by;
    const int g = nx / V;
    if (L.bx == g && 32 % g == 0 && T % 32 == 0) {
        L.warprow = true;
        return;
    }
    if (T >= g) {
        const int rows = std::min(T / g, kXchRows);
        const double busy = (double)rows * g / ((rows * g + 31) / 32 * 32);
        if (B.store == FLB_STORE_F32 || busy >= (V == 4 ? 1.0 : 0.95)) {
            L.rows = rows;
            return;
        }
    }
    L.edgerow = L.by == 1 && g >= 0.95 * ((g + T - 1) / T * T);
}

// The block of whole rows of g threads (g <= 256) that keeps most threads busy:
// the share of its threads that own sites, times the warps an SM holds of it (at
// 128 registers a thread, 512 threads) over 16.  96 wide (g = 24): 96 threads,
// 35.0 GLUPS (FP32, AB) against 29.8 with 128 threads of 32 per row.
inline int row_block(int g)
{
    int best = (g + 31) / 32 * 32;
    double top = 0.0;
    for (int rows = 1; rows <= kXchRows && rows * g <= 256; ++rows) {
        const int T = (rows * g + 31) / 32 * 32;
        const double busy = (double)rows * g / T * (512 / T * T / 512.0);
        if (busy > top + 1e-9) {
            top = busy;
            best = T;
        }
    }
    return best;
}

// Whole rows per block of an FP32 box of a batch, whose blocks of T threads serve
// boxes of every width: T / g rows of g threads where the threads that are left
// over cost less than the whole-row exchange gains over threads packed densely
// over the box (0: packed).  They cost their share of the SM's threads, more so in
// large blocks, of which the SM holds few; the exchange gains most for AA steps
// with four sites per thread, which have the most scalar accesses without it.  The
// line is where both ran equal, 8 boxes of 0.75 M sites, 10 to 34 widths for each T
// (whole rows / packed at a busy share of 0.66, 0.75, 0.84, 0.94):
//   AB V = 4, T 128  0.91 0.98 1.06 1.11   T 256  0.82 0.89 0.94 1.00
//   AB V = 2, T 128  0.93 1.02 1.12 1.20   T 256  0.91 1.00 1.06 1.14
//   AA V = 4, T 128  0.99 1.08 1.15 1.22   T 256  0.92 1.00 1.06 1.14
//   AA V = 2, T 128  0.85 0.93 1.00 1.06   T 256  0.83 0.91 0.96 1.04
// Blocks of one warp gain nothing.  A batch of 264-wide boxes (66 of 128 threads
// busy with whole rows), AB: 29.5 GLUPS with whole rows, 40.8 packed.
inline int batch_rows(int g, int T, int V, bool aa)
{
    if (g > T || T < 64) return 0;
    const int rows = std::min(T / g, kXchRows);
    double least = aa ? (V == 4 ? 0.70 : 0.86) : (V == 4 ? 0.78 : 0.76);
    if (T > 128) least += (T - 128) / 128.0 * (aa ? (V == 4 ? 0.09 : 0.05) : (V == 4 ? 0.17 : 0.05));
    return (double)rows * g / T >= least ? rows : 0;
}

// The shape for what a caller leaves open (sites_per_thread, block_x, block_y; 0 = open).
inline Launch automatic_launch(const LaunchBoxes &B, int sites_per_thread, int block_x, int block_y)
{
    int maxnx = 1;
    for (int nx : B.nx) maxnx = std::max(maxnx, nx);
    const bool f64 = B.store == FLB_STORE_F64;
    Launch L;
    if (B.d2) {
        // warps along x, 256 threads; 4 sites per thread (2 for FP64) when nx allows
        int bx = 32;
        while (bx < maxnx && bx < 128) bx *= 2;
        L.bx = block_x ? block_x : bx;
        L.by = block_y ? block_y : std::max(1, 256 / L.bx);
        L.V = usable_V(B, sites_per_thread ? sites_per_thread : (f64 ? 2 : 4), L.bx, L.by);
        if (L.V == 2 && !f64) L.V = 1;   // the D2Q9 vector kernel has V = 4 (FP64: 2)
        return L;
    }
    int want = sites_per_thread ? sites_per_thread : (f64 ? 2 : 4);
    if (!sites_per_thread) {
        // small boxes: fewer sites per thread until there are threads enough to
        // fill the GPU (~100k: 152 SMs x ~650), measured best for 32^3 and 64^3
        while (want > 1 && B.sites / want < 100000) want /= 2;
    }
    if (f64) want = std::min(want, 2);
    const int sites = (maxnx + want - 1) / want;
    int bx = 32, by = 0;
    while (bx < sites && bx < 128) bx *= 2;
    if (B.nx.size() == 1) {
        int V = want;
        while (maxnx % V != 0) V /= 2;
        const int g = maxnx / V;
        if (V > 1 && g <= 32 && 32 % g == 0) {
            bx = g;          // several rows per warp
        } else if (!block_x && !block_y) {
            by = 1;
            if (V > 1) {
                Launch r;
                r.V = V;
                r.by = 1;
                r.bx = g <= 256 ? row_block(g) : 128;
                set_exchange(B, r);
                // blocks of one row each, of 64 to 160 threads
                for (int nb = (g + 159) / 160; !r.rows && (nb == (g + 159) / 160 || !r.edgerow) && (g + nb - 1) / nb >= 64; ++nb) {
                    r.bx = ((g + nb - 1) / nb + 31) / 32 * 32;
                    set_exchange(B, r);
                }
                bx = r.rows || r.edgerow ? r.bx : 128;
            }
            // FP64 occupies the SM's FP64 unit 64 cycles per warp instruction: one-warp blocks spread a small
            // box over the SMs (16^3: 7.8 us per step, 9.1 with 128 threads; 32^3: 14.0, 16.1)
            else bx = f64 && B.sites < 100000 ? 32 : 128;
        }
    }
    L.bx = block_x ? block_x : bx;
    L.by = block_y ? block_y : (by ? by : std::max(1, 128 / L.bx));
    L.V = usable_V(B, want, L.bx, L.by);
    set_exchange(B, L);
    return L;
}

// What the autotuner times: the shape in use, the automatic shapes for every number
// of sites per thread (whose blocks follow the rows: 96, 160, 32 ... threads), and
// fixed blocks; each shape once.
inline std::vector<Launch> launch_candidates(const LaunchBoxes &B, const Launch &now)
{
    std::vector<Launch> out{now};
    auto add = [&](const Launch &L) {
        for (const Launch &o : out)
            if (o.V == L.V && o.bx == L.bx && o.by == L.by) return;
        out.push_back(L);
    };
    for (int V : {0, 1, 2, 4}) add(automatic_launch(B, V, 0, 0));
    int maxnx = 1;
    for (int nx : B.nx) maxnx = std::max(maxnx, nx);
    const int shapes[9][2] = {{32, 4}, {64, 2}, {64, 4}, {128, 1}, {128, 2}, {256, 1}, {16, 8}, {16, 16}, {32, 8}};
    for (int V : {1, 2, 4}) {
        for (const auto &s : shapes) {
            Launch L;
            L.V = V;
            L.bx = s[0];
            L.by = s[1];
            if (usable_V(B, V, L.bx, L.by) != V) continue;
            // the D2Q9 vector kernel has one width per format
            if (B.d2 && V != 1 && V != (B.store == FLB_STORE_F64 ? 2 : 4)) continue;
            if (L.bx * V > 2 * std::max(32, maxnx)) continue;   // mostly idle threads
            set_exchange(B, L);
            add(L);
        }
    }
    return out;
}

}  // namespace flb
