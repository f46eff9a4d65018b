// lbm_kernels.cuh -- device kernels of liblbm and the host-side launch
// helpers they share.  Population buffers hold post-collision deviations
// f*_a(x, t-1) - w_a rho_ref in the pull convention: the population that
// arrives at x at time t is f*_a(x - e_a, t-1) (Eq. 1 / Eq. 36 streaming).
#pragma once
#include <cuda_runtime.h>
#include <cstddef>
#include <cstdint>

#include "lbm.h"
#include "lbm_device.cuh"
#include "lbm_host.h"
#include "lbm_index.cuh"

namespace lbm {

// FP64 reduction record, one per block of the observe kernel.
struct Partial {
    double mass, row_mid, row0;
    double max_v, max_dv, rho_max, neg_rho_min;
    unsigned status, pad;
};

// Device copy of the lattice observables (mirrors lbm_stats).
struct DevStats {
    double mass, max_v, max_dv, rho_min, rho_max;
    double rho_center, rho_corner, rho_row_mid, rho_row0;
    unsigned status, pad;
};

__device__ __forceinline__ int wrap_any(int v, int n) { int r = v % n; return r < 0 ? r + n : r; }
// x in [0, n): x - 1 and x + 1 with periodic wrap (valid for any n >= 1).
__device__ __forceinline__ int dec1(int x, int n) { return x == 0 ? n - 1 : x - 1; }
__device__ __forceinline__ int inc1(int x, int n) { return x == n - 1 ? 0 : x + 1; }

// Pulled deviations at node (x, y): g_a = f*_a(x - e_a, y - e_a).
template <typename T, typename C>
__device__ __forceinline__ void pull_node(const T* __restrict__ f, int x, int y, int nx, int ny, size_t n, C g[9])
{
    const int xm = dec1(x, nx), xp = inc1(x, nx);
    const int ym = dec1(y, ny), yp = inc1(y, ny);
    const size_t r0 = (size_t)y * nx, rm = (size_t)ym * nx, rp = (size_t)yp * nx;
    g[0] = C(f[0 * n + r0 + x]);
    g[1] = C(f[1 * n + r0 + xm]);
    g[2] = C(f[2 * n + rm + x]);
    g[3] = C(f[3 * n + r0 + xp]);
    g[4] = C(f[4 * n + rp + x]);
    g[5] = C(f[5 * n + rm + xm]);
    g[6] = C(f[6 * n + rm + xp]);
    g[7] = C(f[7 * n + rp + xp]);
    g[8] = C(f[8 * n + rp + xm]);
}

template <typename C>
__device__ __forceinline__ C sum9(const C g[9])
{
    if constexpr (sizeof(C) == sizeof(float))
        return g[0] + moving_sum(g);   // the FP32 collision's density, same order
    else
        return ((g[0] + (g[1] + g[3])) + (g[2] + g[4])) + ((g[5] + g[7]) + (g[6] + g[8]));
}

__device__ __forceinline__ void flag_status(unsigned bad, unsigned* status)
{
    const unsigned w = __reduce_or_sync(0xffffffffu, bad);
    if (w && (threadIdx.x & 31) == 0) atomicOr(status, w);
}

// ---------------------------------------------------------------------------
// Generic fused step, any nx, ny >= 1: a CTA owns a tile of at most 256 nodes,
// one node per thread, and psi also on the ring of nodes around it.  Threads
// [0, w h) take the tile's nodes and the warps after them the ring's, so psi
// of both is evaluated at once from one round of loads; the tile's threads
// keep their pulled populations from there to their collision (which takes F
// from the psi of the tile and ring in shared memory).
//
// What bounds it: in FP64 the FP64 pipe, which takes 64 cycles per warp
// instruction and SM quarter whatever lanes are active; on small FP32
// lattices the latency of one load round.  The tile (plan_tiles) is therefore
// cut to fill every SM quarter evenly, down to one row of 8 nodes, instead of
// a fixed 32 x 8 (a 64 x 64 lattice gave 16 SMs work).  Per step, 32 x 8
// tiles with the pull repeated after the psi pass against this: 64 x 64 FP64
// 14.8 and 7.4 us, 1024 x 1024 FP64 (the 64-thread strips then) 445 and 356,
// 256 x 256 FP32 6.2 and 3.0, 1023 x 1021 FP32 28.9 and 23.1.  Tiles of up to
// 512 nodes gain nothing more (355 us at 1024 x 1024).
//
// Launched as a programmatic dependent of the previous kernel on the stream,
// as the strip step: it touches memory only after griddepcontrol.wait, and
// lets the next step's CTAs be scheduled while this one runs.  A kernel that
// starts so takes no __restrict__ pointers: the qualifier says that nothing
// else writes the memory while the kernel runs, which allows loads through
// the read-only cache and ahead of the wait, when the grid before may still
// be writing it.  The functions called after the wait (step_tile, tile_walk)
// may use it.
// ---------------------------------------------------------------------------
constexpr int GTX = 32, GTY = 8;   // observation tiles

// One tile [x0, x0 + w) x [y0, y0 + h) of an nx x ny lattice: every thread of
// the CTA calls it, after its griddepcontrol.wait.
template <typename T, typename C, int COLL, int FORC>
__device__ __forceinline__ void step_tile(const T* __restrict__ fin, T* __restrict__ fout, int nx, int ny, int x0, int y0,
                                          int w, int h, const Coef<C>& k, C* __restrict__ sp, unsigned& bad)
{
    const size_t n = (size_t)nx * ny;
    const int t = threadIdx.x, W = w + 2;
    const bool own = t < w * h;
    int lx, ly;
    bool live = own;
    if (own) {
        ly = t / w;
        lx = t - ly * w;
    } else {   // the ring: rows -1 and h (w + 2 nodes each), then columns -1 and w
        int r = t - (w * h + 31) / 32 * 32;
        live = r >= 0 && r < 2 * W + 2 * h;
        if (r < 2 * W) {
            ly = r < W ? -1 : h;
            lx = (r < W ? r : r - W) - 1;
        } else {
            r -= 2 * W;
            lx = r < h ? -1 : w;
            ly = r < h ? r : r - h;
        }
    }
    C g[9];
    if (live) {
        const int xs = x0 + lx, ys = y0 + ly;   // one wrap at most: the tile is no larger than the lattice
        pull_node<T, C>(fin, xs < 0 ? nx - 1 : (xs == nx ? 0 : xs), ys < 0 ? ny - 1 : (ys == ny ? 0 : ys), nx, ny, n, g);
        sp[(ly + 1) * W + lx + 1] = psi_of_rho<C>(k.rho_ref + sum9(g), k, bad);
    }
    __syncthreads();
    if (own) {
        const int c = (ly + 1) * W + lx + 1;
        Stencil<C> q{sp[c], sp[c + 1], sp[c + W], sp[c - 1], sp[c - W],
                     sp[c + W + 1], sp[c + W - 1], sp[c - W - 1], sp[c - W + 1]};
        C Fx, Fy, vx, vy, rho;
        force<C>(q, k, Fx, Fy);
        collide<C, COLL, FORC>(g, Fx, Fy, k, vx, vy, rho, q.c);
        bad |= finite_bits<C>(g);
        const size_t o = (size_t)(y0 + ly) * nx + x0 + lx;
#pragma unroll
        for (int a = 0; a < 9; ++a) fout[a * n + o] = T(g[a]);
    }
}

template <typename T, typename C, int COLL, int FORC>
__global__ void __launch_bounds__(kTileThreads)
k_step_generic(const T* fin, T* fout, int nx, int ny, Coef<C> k, unsigned* status)
{
    __shared__ C sp[kTilePsi];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int x0 = int((long long)blockIdx.x * nx / gridDim.x), y0 = int((long long)blockIdx.y * ny / gridDim.y);
    const int w = int((long long)(blockIdx.x + 1) * nx / gridDim.x) - x0;
    const int h = int((long long)(blockIdx.y + 1) * ny / gridDim.y) - y0;
    unsigned bad = 0;
    step_tile<T, C, COLL, FORC>(fin, fout, nx, ny, x0, y0, w, h, k, sp, bad);
    flag_status(bad, status);
}

// ---------------------------------------------------------------------------
// Observation: rho, v = u + F/(2 rho) at time t for every node.
// ---------------------------------------------------------------------------
enum : int { OBS_FIELDS = 1, OBS_REDUCE = 2, OBS_SNAP_CMP = 4, OBS_SNAP_STORE = 8 };

// Velocity snapshot of one node in the compute type (v is computed in it, so
// a float snapshot of the FP32 path loses nothing).
template <typename C> struct VSnapOf;
template <> struct VSnapOf<float> { using type = float2; };
template <> struct VSnapOf<double> { using type = double2; };
template <typename C> using VSnap = typename VSnapOf<C>::type;
__device__ __forceinline__ float2 make_vsnap(float x, float y) { return make_float2(x, y); }
__device__ __forceinline__ double2 make_vsnap(double x, double y) { return make_double2(x, y); }

// rho - rho_ref and v = u + F/(2 rho) of one node from its pulled deviations
// (Eq. 3 and Sec. 3.2), as every observation computes them (FP32: the
// reciprocal Newton-refined).
template <typename C>
__device__ __forceinline__ void node_velocity(const C g[9], C Fx, C Fy, const Coef<C>& k, C& drho, C& vx, C& vy)
{
    C jx, jy;
    moments<C>(g, drho, jx, jy);
    const C rc = k.rho_ref + drho;
    if constexpr (sizeof(C) == sizeof(float)) {
        const float inv = rcp_nr(rc);
        vx = fma_rn(0.5f * Fx, inv, jx * inv);
        vy = fma_rn(0.5f * Fy, inv, jy * inv);
    } else {
        // one division a component (7.4 FP64 instructions), and where j and F/2
        // nearly cancel no error of the size of F/2
        vx = (jx + C(0.5) * Fx) / rc;
        vy = (jy + C(0.5) * Fy) / rc;
    }
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_max(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ float warp_max(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
template <typename C> __device__ __forceinline__ C obs_huge();
template <> __device__ __forceinline__ double obs_huge<double>() { return 1e300; }
template <> __device__ __forceinline__ float obs_huge<float>() { return 1e30f; }

// Observables of a lattice into one FP64 Partial per 32 x 8 tile (fixed-order
// warp shuffles and shared memory: deterministic), for callers that bring
// neither a context nor a workspace (lbm_stats_noalloc).
// The per-node work stays in the compute type C: |v| and the
// density extremes (tracked as max drho and max -drho, then rho = rho_ref +
// drho once per block -- exact, since that sum rounds monotonically in drho)
// are maxima, which are exact in any precision, so only the mass and the two
// probe-row sums need FP64 arithmetic; the row sums are taken only by the
// warps that hold those rows (a warp is one tile row).  This keeps the FP32
// path off the FP64 pipe, which is narrow on this GPU.
template <typename T, typename C>
__global__ void __launch_bounds__(GTX * GTY)
k_observe(const T* __restrict__ fin, int nx, int ny, Coef<C> k, Partial* __restrict__ parts, DevStats* __restrict__ ds)
{
    __shared__ C sp[(GTY + 2) * (GTX + 2)];
    __shared__ double red[6][GTX * GTY / 32];
    const int x0 = blockIdx.x * GTX, y0 = blockIdx.y * GTY;
    const size_t n = (size_t)nx * ny;
    unsigned bad = 0;
    for (int i = threadIdx.x; i < (GTX + 2) * (GTY + 2); i += blockDim.x) {
        const int x = wrap_any(x0 + i % (GTX + 2) - 1, nx);
        const int y = wrap_any(y0 + i / (GTX + 2) - 1, ny);
        C g[9];
        pull_node<T, C>(fin, x, y, nx, ny, n, g);
        sp[i] = psi_of_rho<C>(k.rho_ref + sum9(g), k, bad);
    }
    __syncthreads();
    const int tx = threadIdx.x % GTX, ty = threadIdx.x / GTX;
    const int x = x0 + tx, y = y0 + ty;
    double mass = 0, rho = 0;
    C mv = 0, dmax = -obs_huge<C>(), ndmin = -obs_huge<C>();
    if (x < nx && y < ny) {
        C g[9];
        pull_node<T, C>(fin, x, y, nx, ny, n, g);
        const int W = GTX + 2, c = (ty + 1) * W + tx + 1;
        Stencil<C> q{sp[c], sp[c + 1], sp[c + W], sp[c - 1], sp[c - W],
                     sp[c + W + 1], sp[c + W - 1], sp[c - W - 1], sp[c - W + 1]};
        C Fx, Fy, drho, vx, vy;
        force<C>(q, k, Fx, Fy);
        node_velocity<C>(g, Fx, Fy, k, drho, vx, vy);
        rho = double(k.rho_ref) + double(drho);
        if (!isfinite(drho) || !isfinite(vx) || !isfinite(vy)) bad |= ST_NONFINITE;
        mass = rho;
        mv = sqrt(vx * vx + vy * vy);
        if (isnan(mv)) mv = obs_huge<C>();
        dmax = drho;
        ndmin = -drho;
        if (x == nx / 2 && y == ny / 2) ds->rho_center = rho;
        if (x == 0 && y == 0) ds->rho_corner = rho;
    }
    const unsigned allbad = __reduce_or_sync(0xffffffffu, bad);
    const bool mid_row = y == ny / 2, row_0 = y == 0;      // uniform over the warp
    const C wdmax = warp_max(dmax), wndmin = warp_max(ndmin);
    const double v[6] = {warp_sum(mass), mid_row ? warp_sum(rho) : 0.0, row_0 ? warp_sum(rho) : 0.0, double(warp_max(mv)),
                         double(k.rho_ref) + double(wdmax), -(double(k.rho_ref) + double(-wndmin))};
    __shared__ unsigned sbad;
    if (threadIdx.x == 0) sbad = 0;
    __syncthreads();
    const int wid = threadIdx.x / 32, lane = threadIdx.x % 32;
    if (lane == 0) {
#pragma unroll
        for (int j = 0; j < 6; ++j) red[j][wid] = v[j];
        if (allbad) atomicOr(&sbad, allbad);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        constexpr int NW = GTX * GTY / 32;
        Partial p;
        p.mass = p.row_mid = p.row0 = 0;
        p.max_v = p.rho_max = p.neg_rho_min = -1e300;
        p.max_dv = 0.0;   // (no snapshot to compare with)
        for (int w = 0; w < NW; ++w) {
            p.mass += red[0][w]; p.row_mid += red[1][w]; p.row0 += red[2][w];
            p.max_v = fmax(p.max_v, red[3][w]);
            p.rho_max = fmax(p.rho_max, red[4][w]); p.neg_rho_min = fmax(p.neg_rho_min, red[5][w]);
        }
        p.status = sbad;
        p.pad = 0;
        parts[blockIdx.y * gridDim.x + blockIdx.x] = p;
    }
}

// Fixed-order reduction of the per-block partials into DevStats.
static __global__ void __launch_bounds__(256)
k_reduce_final(const Partial* __restrict__ parts, int nparts, int nx, DevStats* __restrict__ ds)
{
    __shared__ double red[7][256];
    __shared__ unsigned sbad[256];
    double v[7] = {0, 0, 0, -1e300, -1e300, -1e300, -1e300};
    unsigned bad = 0;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x) {
        const Partial p = parts[i];
        v[0] += p.mass; v[1] += p.row_mid; v[2] += p.row0;
        v[3] = fmax(v[3], p.max_v); v[4] = fmax(v[4], p.max_dv);
        v[5] = fmax(v[5], p.rho_max); v[6] = fmax(v[6], p.neg_rho_min);
        bad |= p.status;
    }
    for (int j = 0; j < 7; ++j) red[j][threadIdx.x] = v[j];
    sbad[threadIdx.x] = bad;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            const int o = threadIdx.x + s;
            red[0][threadIdx.x] += red[0][o]; red[1][threadIdx.x] += red[1][o]; red[2][threadIdx.x] += red[2][o];
            for (int j = 3; j < 7; ++j) red[j][threadIdx.x] = fmax(red[j][threadIdx.x], red[j][o]);
            sbad[threadIdx.x] |= sbad[o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        ds->mass = red[0][0];
        ds->rho_row_mid = red[1][0] / nx;
        ds->rho_row0 = red[2][0] / nx;
        ds->max_v = red[3][0];
        ds->max_dv = red[4][0];
        ds->rho_max = red[5][0];
        ds->rho_min = -red[6][0];
        ds->status = sbad[0];
    }
}

// ---------------------------------------------------------------------------
// State conversion between post-streaming populations f_a(x, t) (FP64, the
// user-facing form) and the stored pull-convention deviations
// f*_a(x, t-1) - w_a rho_ref = f_a(x + e_a, t) - w_a rho_ref.
// ---------------------------------------------------------------------------
// A start at rest, f_a = w_a rho0, as stored values in one pass: the thread of
// a node writes its population of direction a to the node that stores it,
// x - e_a (a warp's stores stay contiguous).  FP32: w_a float(rho0 - rho_ref),
// so one FP64 subtraction a node.  Bound by HBM, 8 B read and 36 B (FP64 72 B)
// written per node; in two passes through an array of deviations, each node
// found by a 64-bit division, 4096 x 4096 took 200 us in FP32, now 144.  One
// linear walk over the nodes: on a grid of 256-column blocks by rows, narrow
// lattices kept 1 to 16 of 256 threads busy (4 x 262144: 43 us, now 11; the two
// passes 19) and column indices overflowed near 2^31 columns.
template <typename T>
__global__ void __launch_bounds__(256)
k_init_rest(const double* __restrict__ rho0, T* __restrict__ fs, int nx, int ny, double rho_ref)
{
    const unsigned n = unsigned(nx) * unsigned(ny);
    for (NodeWalk w(blockIdx.x * 256 + threadIdx.x, gridDim.x * 256, nx); w.id < n; w.next()) {
        const int x = int(w.x), y = int(w.y), xl = dec1(x, nx), xr = inc1(x, nx);
        const size_t row = (size_t)y * nx, rd = (size_t)dec1(y, ny) * nx, ru = (size_t)inc1(y, ny) * nx;
        const double r = rho0[w.id];
        const float d = float(r - rho_ref);
#pragma unroll
        for (int a = 0; a < 9; ++a) {
            const size_t at = (ey(a) > 0 ? rd : (ey(a) < 0 ? ru : row)) + (ex(a) > 0 ? xl : (ex(a) < 0 ? xr : x));
            if constexpr (sizeof(T) == sizeof(float)) fs[(size_t)a * n + at] = wt<float>(a) * d;
            else fs[(size_t)a * n + at] = T(wt<double>(a) * r - wt<double>(a) * rho_ref);
        }
    }
}

// One plane a: stored <- post-streaming (dir = +1) or post-streaming <- stored (dir = -1).
template <typename T>
__global__ void k_plane_convert(T* __restrict__ fs, double* __restrict__ plane, int a, int nx, int ny,
                                double rho_ref, int to_stored)
{
    const size_t n = (size_t)nx * ny;
    const double w = wt<double>(a);
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const int x = int(i % nx), y = int(i / nx);
        if (to_stored) {   // fs_a(x) = f_a(x + e_a)
            const int xs = ex(a) > 0 ? inc1(x, nx) : (ex(a) < 0 ? dec1(x, nx) : x);
            const int ys = ey(a) > 0 ? inc1(y, ny) : (ey(a) < 0 ? dec1(y, ny) : y);
            fs[a * n + i] = T(plane[(size_t)ys * nx + xs] - w * rho_ref);
        } else {           // f_a(x) = fs_a(x - e_a)
            const int xs = ex(a) > 0 ? dec1(x, nx) : (ex(a) < 0 ? inc1(x, nx) : x);
            const int ys = ey(a) > 0 ? dec1(y, ny) : (ey(a) < 0 ? inc1(y, ny) : y);
            plane[i] = double(fs[a * n + (size_t)ys * nx + xs]) + w * rho_ref;
        }
    }
}

// The observation of a lattice (lbm_observe.cu): mode of OBS_ flags; with
// OBS_REDUCE the per-CTA partials (parts, at least as many as 32 x 8 tiles)
// are reduced in the same launch by the last CTA to finish, in a fixed order,
// into ds (ticket: a device counter that is 0 between launches).  vsnap holds
// VSnap<C> of the precision's compute type.
int observe_launch(const lbm_params* p, const void* f, int mode, double* rho, double* vx, double* vy, void* vsnap,
                   Partial* parts, unsigned* ticket, DevStats* ds, const unsigned* status, int nsm, cudaStream_t s);

}  // namespace lbm
