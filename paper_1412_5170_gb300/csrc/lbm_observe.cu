// lbm_observe.cu -- the lattice observables (rho, v = u + F/(2 rho) at time t,
// FP64 mass, max |v|, max |v - v_snap|, density extremes and probes, status)
// with the walks of the time step -- the strip walk (lbm_strip.cuh) of large
// FP32 lattices, the walk of tiles (lbm_tilewalk.cuh) of all others: the same row
// copies or loads, psi and pulled populations, but each node is observed
// instead of collided, so its populations are read from HBM once (36 B per
// node in FP32, 72 B in FP64) and nothing is written unless the moment fields
// or the velocity snapshot are asked for.
//
// With OBS_REDUCE every CTA leaves one FP64 Partial, and the last CTA to
// finish (a ticket counter) reduces all of them in a fixed order into the
// DevStats record in the same launch: the result is the same bit for bit
// from run to run.
#include <algorithm>

#include "lbm.h"
#include "lbm_host.h"
#include "lbm_strip.cuh"
#include "lbm_tilewalk.cuh"

namespace lbm {
namespace {

// Running reductions of one thread, and the probe rows' sums.  The mass is
// N rho_ref plus the sum of the deviations drho, in FP64.  PAIR (strips of FP32
// deviations): a float pair (sum, error) kept by Knuth's TwoSum, which
// carries every addition's rounding into the error term (six FP32
// additions a node instead of a conversion and an addition on this GPU's
// narrow FP64 pipe), converted to FP64 once per thread.  The walks of tiles,
// which also serve widths whose sums were never pairs, hide one FP64 addition
// a node behind its other 400 instructions.  The maxima are taken
// on |v|^2 and |v - v_snap|^2 in the compute type (exact) and rooted once per
// CTA.
template <typename C, bool PAIR>
struct ObsAcc {
    double dmass = 0.0, row_mid = 0.0, row0 = 0.0;
    C mv2 = C(0), mdv2 = C(0), dmax = -obs_huge<C>(), ndmin = -obs_huge<C>();
    float ms = 0.f, me = 0.f;   // PAIR: running sum of drho and its accumulated rounding

    __device__ __forceinline__ void node(C d, C vx, C vy)
    {
        const C s2 = vx * vx + vy * vy;
        mv2 = (s2 > mv2 || s2 != s2) ? s2 : mv2;      // NaN wins (reported as huge)
        dmax = d > dmax ? d : dmax;
        ndmin = -d > ndmin ? -d : ndmin;
        if constexpr (PAIR) {
            const float t = ms + d;
            const float bp = t - ms;
            me += (ms - (t - bp)) + (d - bp);
            ms = t;
        } else {
            dmass += double(d);
        }
    }
    __device__ __forceinline__ void change(C dx, C dy)
    {
        const C d2 = dx * dx + dy * dy;
        mdv2 = (d2 > mdv2 || d2 != d2) ? d2 : mdv2;
    }
};
struct ObsOut {
    int mode, nx, ny;
    double* __restrict__ rho_o;
    double* __restrict__ vx_o;
    double* __restrict__ vy_o;
    DevStats* __restrict__ ds;   // null without OBS_REDUCE
};

// Strip walk: each chunk row, four nodes a thread.
template <typename T, typename C>
struct ObsRow {
    ObsOut to;
    VSnap<C>* __restrict__ vsnap;
    ObsAcc<C, sizeof(C) == sizeof(float)> acc;
    __device__ __forceinline__ void operator()(int y, int x, bool active, C (&gc)[9][4], const C (&rm)[6],
                                               const C (&r0)[6], const C (&rp)[6], const Coef<C>& k,
                                               unsigned& bad)
    {
        if (!active) return;
        const int mode = to.mode, nx = to.nx, ny = to.ny;
        DevStats* const ds = to.ds;
        C d4[4], vx4[4], vy4[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            Stencil<C> q{r0[j + 1], r0[j + 2], rp[j + 1], r0[j], rm[j + 1], rp[j + 2], rp[j], rm[j], rm[j + 2]};
            C Fx, Fy, g[9];
            force<C>(q, k, Fx, Fy);
#pragma unroll
            for (int a = 0; a < 9; ++a) g[a] = gc[a][j];
            node_velocity<C>(g, Fx, Fy, k, d4[j], vx4[j], vy4[j]);
            acc.node(d4[j], vx4[j], vy4[j]);
        }
        if (!isfinite(acc.dmax) || !isfinite(acc.ndmin) || !isfinite(acc.mv2)) bad |= ST_NONFINITE;
        if (y == ny / 2 || y == 0 || (mode & OBS_FIELDS)) {
            double rho4[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) rho4[j] = double(k.rho_ref) + double(d4[j]);
            if (y == ny / 2) acc.row_mid += (rho4[0] + rho4[1]) + (rho4[2] + rho4[3]);
            if (y == 0) acc.row0 += (rho4[0] + rho4[1]) + (rho4[2] + rho4[3]);
            if (ds && y == ny / 2 && x <= nx / 2 && nx / 2 < x + 4) {
                const int j = nx / 2 - x;
                ds->rho_center = j == 0 ? rho4[0] : (j == 1 ? rho4[1] : (j == 2 ? rho4[2] : rho4[3]));
            }
            if (ds && y == 0 && x == 0) ds->rho_corner = rho4[0];
            if (mode & OBS_FIELDS) {
                const size_t o = (size_t)y * nx + x;   // x % 4 == 0 and nx % 4 == 0: 4-node aligned
                stg4(to.rho_o + o, rho4[0], rho4[1], rho4[2], rho4[3]);
                stg4(to.vx_o + o, double(vx4[0]), double(vx4[1]), double(vx4[2]), double(vx4[3]));
                stg4(to.vy_o + o, double(vy4[0]), double(vy4[1]), double(vy4[2]), double(vy4[3]));
            }
        }
        const size_t o = (size_t)y * nx + x;
        if (mode & OBS_SNAP_CMP) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const VSnap<C> sv = vsnap[o + j];
                acc.change(vx4[j] - C(sv.x), vy4[j] - C(sv.y));
            }
        }
        if (mode & OBS_SNAP_STORE) {
#pragma unroll
            for (int j = 0; j < 4; ++j) vsnap[o + j] = make_vsnap(vx4[j], vy4[j]);
        }
    }
};

// Walk of tiles: one node a thread, a warp one row of the strip.
template <typename C>
struct ObsNode {
    ObsOut to;
    VSnap<C>* __restrict__ vsnap;
    double* __restrict__ rows;   // shared: sums of rho over the strip's part of rows ny/2 and 0
    int w;                       // the strip's width: lanes 0 .. w - 1 hold its columns
    ObsAcc<C, false> acc;

    __device__ __forceinline__ void operator()(int y, int x, C (&g)[9], const Stencil<C>& q, const Coef<C>& k,
                                               unsigned& bad)
    {
        const int mode = to.mode;
        const size_t o = (size_t)y * to.nx + x;
        VSnap<C> sv{};
        if (mode & OBS_SNAP_CMP) sv = vsnap[o];   // fetched under the node's arithmetic
        C Fx, Fy, d, vx, vy;
        force<C>(q, k, Fx, Fy);
        node_velocity<C>(g, Fx, Fy, k, d, vx, vy);
        acc.node(d, vx, vy);
        if (!isfinite(d) || !isfinite(acc.mv2)) bad |= ST_NONFINITE;
        const bool mid = y == to.ny / 2;
        if (mid || y == 0 || (mode & OBS_FIELDS)) {   // (uniform over the warp)
            const double rho = double(k.rho_ref) + double(d);
            if (mid || y == 0) {
                const unsigned lanes = w == 32 ? 0xffffffffu : (1u << w) - 1u;
                double s = 0.0;
                for (int i = 0; i < w; ++i) s += __shfl_sync(lanes, rho, i);
                if ((threadIdx.x & 31) == 0) {
                    if (mid) rows[0] = s;
                    if (y == 0) rows[1] = s;
                }
                if (to.ds && mid && x == to.nx / 2) to.ds->rho_center = rho;
                if (to.ds && y == 0 && x == 0) to.ds->rho_corner = rho;
            }
            if (mode & OBS_FIELDS) {
                to.rho_o[o] = rho;
                to.vx_o[o] = double(vx);
                to.vy_o[o] = double(vy);
            }
        }
        if (mode & OBS_SNAP_CMP) acc.change(vx - C(sv.x), vy - C(sv.y));
        if (mode & OBS_SNAP_STORE) vsnap[o] = make_vsnap(vx, vy);
    }
};

// max over a warp of a squared magnitude, then its root (NaN -> huge)
template <typename C>
__device__ __forceinline__ double warp_max_root(C v2)
{
    const C w = warp_max(v2 != v2 ? obs_huge<C>() : v2);
    return double(sqrt(w));
}

// The CTA's partial from its threads' reductions (warp shuffles, then the
// warps in order), and in the last CTA to get here the fold of all partials.
// red [7 NW], sbad [NW] and last are shared memory.
template <typename C, int NT, bool PAIR>
__device__ __forceinline__ void reduce_and_fold(ObsAcc<C, PAIR>& acc, unsigned bad, double cta_nodes, const Coef<C>& k, int nx,
                                                double* red, unsigned* sbad, unsigned* last,
                                                Partial* __restrict__ parts, unsigned* __restrict__ ticket,
                                                DevStats* __restrict__ ds, const unsigned* __restrict__ status)
{
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if constexpr (PAIR) acc.dmass = double(acc.ms) + double(acc.me);
    double v[7] = {warp_sum(acc.dmass), warp_sum(acc.row_mid), warp_sum(acc.row0), warp_max_root(acc.mv2),
                   warp_max_root(acc.mdv2), 0.0, 0.0};
    const C wdmax = warp_max(acc.dmax), wndmin = warp_max(acc.ndmin);
    v[5] = double(k.rho_ref) + double(wdmax);
    v[6] = -(double(k.rho_ref) + double(-wndmin));
    const unsigned wbad = __reduce_or_sync(0xffffffffu, bad);
    if (lane == 0) {
#pragma unroll
        for (int j = 0; j < 7; ++j) red[j * NW + wid] = v[j];
        sbad[wid] = wbad;
    }
    __syncthreads();
    const unsigned nparts = gridDim.x * gridDim.y;
    if (threadIdx.x == 0) {
        Partial p;
        p.mass = p.row_mid = p.row0 = 0;
        p.max_v = p.max_dv = p.rho_max = p.neg_rho_min = -1e300;
        p.status = 0;
        p.mass = cta_nodes * double(k.rho_ref);
        for (int w = 0; w < NW; ++w) {
            p.mass += red[0 * NW + w]; p.row_mid += red[1 * NW + w]; p.row0 += red[2 * NW + w];
            p.max_v = fmax(p.max_v, red[3 * NW + w]); p.max_dv = fmax(p.max_dv, red[4 * NW + w]);
            p.rho_max = fmax(p.rho_max, red[5 * NW + w]); p.neg_rho_min = fmax(p.neg_rho_min, red[6 * NW + w]);
            p.status |= sbad[w];
        }
        p.pad = 0;
        parts[blockIdx.y * gridDim.x + blockIdx.x] = p;
        __threadfence();
        *last = atomicAdd(ticket, 1u) == nparts - 1;
    }
    __syncthreads();
    if (!*last) return;

    // The last CTA: every partial is written and fenced; fold them in a fixed
    // order (thread t takes t, t + NT, ...; then the warps; then thread 0).
    __threadfence();
    double a[7] = {0, 0, 0, -1e300, -1e300, -1e300, -1e300};
    unsigned b = 0;
    for (unsigned i = threadIdx.x; i < nparts; i += NT) {
        const Partial* q = parts + i;
        a[0] += __ldcg(&q->mass); a[1] += __ldcg(&q->row_mid); a[2] += __ldcg(&q->row0);
        a[3] = fmax(a[3], __ldcg(&q->max_v)); a[4] = fmax(a[4], __ldcg(&q->max_dv));
        a[5] = fmax(a[5], __ldcg(&q->rho_max)); a[6] = fmax(a[6], __ldcg(&q->neg_rho_min));
        b |= __ldcg(&q->status);
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) a[j] = warp_sum(a[j]);
#pragma unroll
    for (int j = 3; j < 7; ++j) a[j] = warp_max(a[j]);
    b = __reduce_or_sync(0xffffffffu, b);
    __syncthreads();
    if (lane == 0) {
#pragma unroll
        for (int j = 0; j < 7; ++j) red[j * NW + wid] = a[j];
        sbad[wid] = b;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double f[7] = {0, 0, 0, -1e300, -1e300, -1e300, -1e300};
        unsigned fb = status ? *status : 0u;
        for (int w = 0; w < NW; ++w) {
            for (int j = 0; j < 3; ++j) f[j] += red[j * NW + w];
            for (int j = 3; j < 7; ++j) f[j] = fmax(f[j], red[j * NW + w]);
            fb |= sbad[w];
        }
        ds->mass = f[0];
        ds->rho_row_mid = f[1] / nx;
        ds->rho_row0 = f[2] / nx;
        ds->max_v = f[3];
        ds->max_dv = f[4];
        ds->rho_max = f[5];
        ds->rho_min = -f[6];
        ds->status = fb;
        *ticket = 0;   // ready for the next launch
    }
}

// One CTA per (strip, row chunk), as the step kernel.  Every CTA reaches the
// reduction, whatever happened to its walk (a misaligned buffer, an empty
// chunk, a stage wait that gave up), so the ticket always completes.
template <typename T, typename C, int NT, int NS, int MINB>
__global__ void __launch_bounds__(NT, MINB)
k_observe_strip(const T* __restrict__ fin, int nx, int ny, int nchunks, Coef<C> k, int mode,
                double* __restrict__ rho_o, double* __restrict__ vx_o, double* __restrict__ vy_o,
                VSnap<C>* __restrict__ vsnap, Partial* __restrict__ parts, unsigned* __restrict__ ticket,
                DevStats* __restrict__ ds, const unsigned* __restrict__ status)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const StripSmem<T, C, NT, NS> sm(smem);
    ObsRow<T, C> row{{mode, nx, ny, rho_o, vx_o, vy_o, (mode & OBS_REDUCE) ? ds : nullptr}, vsnap, {}};
    // (only nodes of this CTA's rows enter the sums; N rho_ref is added to the mass per CTA below)
    unsigned bad = 0;
    const int x0 = blockIdx.x * (4 * NT);
    const int y0 = int((long long)blockIdx.y * ny / nchunks);
    const int y1 = int((long long)(blockIdx.y + 1) * ny / nchunks);
    if (!staged_alignment_ok(smem, fin, fin)) {
        bad |= ST_ALIGN;
    } else if (y1 > y0) {
        strip_init_barriers(sm);
        unsigned G = 0;
        strip_walk<T, C, NT, NS, true, true, true>(fin, nx, ny, x0, y0, y1, (blockIdx.y & 1) != 0, k, sm, G, bad,
                                                    row);
    }
    if (!(mode & OBS_REDUCE)) return;

    __syncthreads();   // the stages are free now
    constexpr int NW = NT / 32;
    double* red = reinterpret_cast<double*>(smem);               // [7][NW]
    unsigned* sbad = reinterpret_cast<unsigned*>(red + 7 * NW);  // [NW], then the last-CTA flag
    // (no static shared memory: it would move the dynamic region off the
    // alignment the bulk copies need)
    const double cta_nodes = double(y1 > y0 ? y1 - y0 : 0) * double(min(4 * NT, nx - x0));
    reduce_and_fold<C, NT>(row.acc, bad, cta_nodes, k, nx, red, sbad, sbad + NW, parts, ticket, ds, status);
}

// The same with the walk of tiles: one CTA per (32-column strip, chunk of `rows` rows).
template <typename T, typename C, int CTAS>
__global__ void __launch_bounds__(kWalkThreads, CTAS)
k_observe_walk(const T* __restrict__ fin, int nx, int ny, int rows, Coef<C> k, int mode,
               double* __restrict__ rho_o, double* __restrict__ vx_o, double* __restrict__ vy_o,
               VSnap<C>* __restrict__ vsnap, Partial* __restrict__ parts, unsigned* __restrict__ ticket,
               DevStats* __restrict__ ds, const unsigned* __restrict__ status)
{
    constexpr int NW = kWalkThreads / 32;
    __shared__ WalkPsi<C> sm;
    __shared__ double red[7 * NW], row_sums[2];
    __shared__ unsigned sbad[NW], last;
    const RowChunk c = row_chunk(blockIdx.y, rows, ny);
    const int x0 = blockIdx.x * kWalkW, w = min(kWalkW, nx - x0);
    if (threadIdx.x < 2) row_sums[threadIdx.x] = 0.0;   // (the walk's barriers come before any row's sum)
    ObsNode<C> node{{mode, nx, ny, rho_o, vx_o, vy_o, (mode & OBS_REDUCE) ? ds : nullptr}, vsnap, row_sums, w, {}};
    unsigned bad = 0;
    tile_walk<T, C>(fin, nx, ny, x0, w, c.y0, c.y1, k, sm, bad, node);
    if (!(mode & OBS_REDUCE)) return;
    __syncthreads();
    if (threadIdx.x == 0) {
        node.acc.row_mid = row_sums[0];
        node.acc.row0 = row_sums[1];
    }
    reduce_and_fold<C, kWalkThreads>(node.acc, bad, double(c.y1 - c.y0) * double(w), k, nx, red, sbad, &last, parts, ticket,
                                     ds, status);
}

template <typename T, typename C, int NT, int NS, int MINB>
int launch_strip(const lbm_params* p, const void* f, int mode, double* rho, double* vx, double* vy, void* vsnap,
           Partial* parts, unsigned* ticket, DevStats* ds, const unsigned* status, cudaStream_t s)
{
    constexpr size_t smem = strip_smem<T, C, NT, NS>();
    static_assert(smem >= (7 * sizeof(double) + sizeof(unsigned)) * (NT / 32) + sizeof(unsigned), "reduction scratch");
    auto kern = k_observe_strip<T, C, NT, NS, MINB>;
    static int per_sm = 0, nsm = 0;   // per instantiation (one device per process)
    if (per_sm == 0) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
            return LBM_E_CUDA;
        int dev = 0, occ = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, NT, smem) != cudaSuccess || occ < 1) occ = 1;
        per_sm = occ;
    }
    const int W = 4 * NT;
    const int nstrips = (p->nx + W - 1) / W;
    int nchunks = std::max(1, (nsm * per_sm) / nstrips);
    nchunks = std::min(nchunks, std::max(1, p->ny / 16));
    kern<<<dim3(nstrips, nchunks), NT, smem, s>>>((const T*)f, p->nx, p->ny, nchunks, make_coef<C>(*p), mode, rho,
                                                  vx, vy, (VSnap<C>*)vsnap, parts, ticket, ds, status);
    return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_E_CUDA;
}

template <typename T, typename C, int CTAS>
int launch_walk(const lbm_params* p, const void* f, int mode, double* rho, double* vx, double* vy, void* vsnap,
                Partial* parts, unsigned* ticket, DevStats* ds, const unsigned* status, int nsm, cudaStream_t s)
{
    const WalkPlan w = plan_walk(p->nx, p->ny, nsm, CTAS);
    k_observe_walk<T, C, CTAS><<<dim3(w.sx, w.sy), kWalkThreads, 0, s>>>(
        (const T*)f, p->nx, p->ny, w.rows, make_coef<C>(*p), mode, rho, vx, vy, (VSnap<C>*)vsnap, parts, ticket, ds, status);
    return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_E_CUDA;
}

}  // namespace

// FP32 from 3 * 2^19 nodes (nx % 4 == 0): the strip walk, whose bulk copies
// keep more of a large lattice in flight; everything else: walks of tiles,
// which spread over more CTAs and take any width.  lbm_stats, walk of tiles
// and strip walk: 64 x 64 37 and 72 us (FP64 50 and 370), 512 x 512 50 and 73
// (FP64 124 and 358), 1024 x 1024 52 and 74 (FP64 353 and 385), 512 x 4096
// 108 and 76, 1536 x 1536 112 and 80, 4096 x 4096 301 and 188 (FP64 from
// 1536 x 1536 on within 1 % of each other).  Strips of 512 columns, four CTAs
// of 128 threads an SM, the left halo's psi off the copying warp: with three
// lattices in turn and snapshots 75.8 us at 1536 x 1536 and 212.2 at
// 4096 x 4096; 1024 columns take 89.9 and 224.6, 2048 columns 99.8 and 249.6.
constexpr long long kObsStripNodes = 3 << 19;

int observe_launch(const lbm_params* p, const void* f, int mode, double* rho, double* vx, double* vy, void* vsnap,
                   Partial* parts, unsigned* ticket, DevStats* ds, const unsigned* status, int nsm, cudaStream_t s)
{
    if (p->precision == LBM_FP64)
        return launch_walk<double, double, 2>(p, f, mode, rho, vx, vy, vsnap, parts, ticket, ds, status, nsm, s);
    if (lbm_strip_supported(p) && (long long)p->nx * p->ny >= kObsStripNodes)
        return launch_strip<float, float, 128, 2, 4>(p, f, mode, rho, vx, vy, vsnap, parts, ticket, ds, status, s);
    return launch_walk<float, float, kWalkCtas>(p, f, mode, rho, vx, vy, vsnap, parts, ticket, ds, status, nsm, s);
}

}  // namespace lbm
