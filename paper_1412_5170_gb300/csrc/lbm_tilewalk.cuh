// lbm_tilewalk.cuh -- the FP32 step as a walk of 32 x 8 tiles down a strip of
// 32 columns, one node per thread, for lattices of any width (plain 32-bit
// loads: no alignment of rows is needed, which the strip walks' 16-byte
// copies take for granted).
//
// Eight warps hold the tile's rows, two more the nodes to its left, right and
// below whose psi the force needs; the psi above is the last row of the tile
// before.  Each thread loads its nine pulled values of the next tile before
// it collides the current one, so a CTA always has a tile of loads in flight;
// a grid of separate tiles (the generic step) waits out the memory latency
// once per tile instead.  One barrier per tile: psi is double-buffered.  Per
// step, separate tiles and this (MRT): 384 x 384 6.1 and 4.7 us, 1023 x 1021
// 22.9 and 19.4, 2047 x 2049 85.4 and 68.8, 4096 x 4096 335 and 252 (the strip
// walks 211); 256 sweep instances (25 M nodes) 479 and 398 (the one-warp strip
// walk 480).  What bounds it is issue: 76 to 79 % of the slots at 2047 x 2049,
// with 471 (MRT) or 529 (BGK) instructions a node.
#pragma once
#include <cuda_runtime.h>

#include "lbm_kernels.cuh"

namespace lbm {

constexpr int kWalkW = 32, kWalkH = 8, kWalkThreads = 32 * (kWalkH + 2);
constexpr int kWalkRow = kWalkW + 2;
constexpr int kWalkCtas = 4;   // per SM: 48 registers a thread

template <typename C>
struct WalkPsi { C p[2][(kWalkH + 2) * kWalkRow]; };

// The time step of one node (x, y) from its pulled populations and the psi
// stencil around it.
template <typename T, typename C, int COLL, int FORC>
struct StepNode {
    T* __restrict__ fout;
    int nx;
    size_t n;
    __device__ __forceinline__ void operator()(int y, int x, C (&g)[9], const Stencil<C>& q, const Coef<C>& k,
                                               unsigned& bad) const
    {
        C Fx, Fy, vx, vy, rho;
        force<C>(q, k, Fx, Fy);
        collide<C, COLL, FORC>(g, Fx, Fy, k, vx, vy, rho, q.c);
        if constexpr (sizeof(C) == sizeof(float)) {
            if (!isfinite(g[0])) bad |= ST_NONFINITE;   // g0 closes on all others
        } else {
            bad |= finite_bits<C>(g);
        }
        T* o = fout + (size_t)y * nx + x;
#pragma unroll
        for (int a = 0; a < 9; ++a) o[a * n] = T(g[a]);
    }
};

// Columns [x0, x0 + w) with w <= 32, rows [y0, y1) of an nx x ny lattice, each
// node handed to `node` once; all kWalkThreads threads call it.
template <typename T, typename C, class Node>
__device__ __forceinline__ void tile_walk(const T* __restrict__ fin, int nx, int ny, int x0, int w, int y0, int y1,
                                          const Coef<C>& k, WalkPsi<C>& sm, unsigned& bad, Node& node)
{
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const size_t n = (size_t)nx * ny;
    const bool mine = wid < kWalkH;
    // ring threads: the row below (w + 2 nodes from column -1 on), then the columns -1 and w of the tile's rows
    const int r = t - 32 * kWalkH;
    const bool below = !mine && r < w + 2;
    const int side = r - (w + 2);   // 0 .. 15: row side / 2 of the left (even) or right (odd) column
    const int lx = mine ? lane : (below ? r - 1 : (side & 1 ? w : -1));
    const bool used = mine ? lane < w : (below || side < 2 * kWalkH);
    // (idle lanes of a ragged strip: any column; x0 + lx itself may exceed 2^31 - 1 there)
    const int xs = lx < -x0 ? nx - 1 : (lx >= nx - x0 ? 0 : x0 + lx);
    const int xm = dec1(xs, nx), xp = inc1(xs, nx);
    // row of this thread's node in a tile of h rows
    auto row_of = [&](int h) { return mine ? wid : (below ? h : side >> 1); };
    auto live_in = [&](int h) { return used && (below || row_of(h) < h); };
    auto load = [&](int y, C (&g)[9]) {
        const int ys = y < 0 ? ny - 1 : (y >= ny ? y - ny : y);
        const size_t r0 = (size_t)ys * nx, rm = (size_t)dec1(ys, ny) * nx, rp = (size_t)inc1(ys, ny) * nx;
        g[0] = C(fin[0 * n + r0 + xs]);
        g[1] = C(fin[1 * n + r0 + xm]);
        g[2] = C(fin[2 * n + rm + xs]);
        g[3] = C(fin[3 * n + r0 + xp]);
        g[4] = C(fin[4 * n + rp + xs]);
        g[5] = C(fin[5 * n + rm + xm]);
        g[6] = C(fin[6 * n + rm + xp]);
        g[7] = C(fin[7 * n + rp + xp]);
        g[8] = C(fin[8 * n + rp + xm]);
    };

    C gA[9], gB[9];
    // the row above the first tile
    if (below) {
        load(y0 - 1, gA);
        sm.p[0][lx + 1] = psi_of_rho<C>(k.rho_ref + sum9(gA), k, bad);
    }
    int h = min(kWalkH, y1 - y0);
    if (live_in(h)) load(y0 + row_of(h), gA);

    auto body = [&](int y, int buf, C (&g)[9], C (&gn)[9]) {
        C* p = sm.p[buf];
        const int ly = row_of(h);
        if (live_in(h)) p[(ly + 1) * kWalkRow + lx + 1] = psi_of_rho<C>(k.rho_ref + sum9(g), k, bad);
        const int hn = min(kWalkH, y1 - y - h);
        if (hn > 0 && live_in(hn)) load(y + h + row_of(hn), gn);   // the next tile, in flight from here
        __syncthreads();
        if (mine && lane < w && ly < h) {
            const int c = (ly + 1) * kWalkRow + lane + 1;
            const Stencil<C> q{p[c], p[c + 1], p[c + kWalkRow], p[c - 1], p[c - kWalkRow],
                               p[c + kWalkRow + 1], p[c + kWalkRow - 1], p[c - kWalkRow - 1], p[c - kWalkRow + 1]};
            node(y + ly, x0 + lane, g, q, k, bad);
        } else if (below) {
            sm.p[buf ^ 1][lx + 1] = p[h * kWalkRow + lx + 1];   // the last row's psi: above the next tile
        }
        h = hn;
    };
    walk_tiles<kWalkH>(y0, y1, [&](int y) { body(y, 0, gA, gB); }, [&](int y) { body(y, 1, gB, gA); });
}

// One lattice: grid (32-column strips, chunks of `rows` rows).
template <int COLL, int FORC>
__global__ void __launch_bounds__(kWalkThreads, kWalkCtas)
k_step_walk(const float* fin, float* fout, int nx, int ny, int rows, Coef<float> k, unsigned* status)
{
    __shared__ WalkPsi<float> sm;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int x0 = blockIdx.x * kWalkW;
    const RowChunk c = row_chunk(blockIdx.y, rows, ny);
    unsigned bad = 0;
    StepNode<float, float, COLL, FORC> node{fout, nx, (size_t)nx * ny};
    tile_walk<float, float>(fin, nx, ny, x0, min(kWalkW, nx - x0), c.y0, c.y1, k, sm, bad, node);
    flag_status(bad, status);
}

}  // namespace lbm
