// lbm_observe.cu -- the lattice observables (rho, v = u + F/(2 rho) at time t,
// FP64 mass, max |v|, max |v - v_snap|, density extremes and probes, status)
// with the walks of the time step -- the strip walk (lbm_strip.cuh) of large
// FP32 lattices, the walk of tiles (lbm_tilewalk.cuh) of all others -- and the
// moment fields alone on separate tiles: the same row copies or loads, psi and
// pulled populations, but each node is observed instead of collided, so its
// populations are read from HBM once (36 B per node in FP32, 72 B in FP64) and
// nothing is written unless the moment fields or the velocity snapshot are
// asked for.
//
// With OBS_REDUCE every CTA leaves one FP64 Partial, and the last CTA to
// finish (a ticket counter) reduces all of them in a fixed order into the
// DevStats record in the same launch: the result is the same bit for bit
// from run to run.
#include <algorithm>
#include <climits>
#include <cstddef>

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
    int mode, nx, ny;
    DevStats* __restrict__ ds;
    VSnap<C>* __restrict__ vsnap;
    ObsAcc<C, false> acc;

    __device__ __forceinline__ void operator()(int y, int x, C (&g)[9], const Stencil<C>& q, const Coef<C>& k,
                                               unsigned& bad)
    {
        const size_t o = (size_t)y * nx + x;
        VSnap<C> sv{};
        if (mode & OBS_SNAP_CMP) sv = vsnap[o];   // fetched under the node's arithmetic
        C Fx, Fy, d, vx, vy;
        force<C>(q, k, Fx, Fy);
        node_velocity<C>(g, Fx, Fy, k, d, vx, vy);
        acc.node(d, vx, vy);
        if (!isfinite(d) || !isfinite(acc.mv2)) bad |= ST_NONFINITE;
        const bool mid = y == ny / 2;
        if (mid || y == 0) {   // (uniform over the warp)
            const double rho = double(k.rho_ref) + double(d);
            if (mid) acc.row_mid += rho;
            if (y == 0) acc.row0 += rho;
            if (mid && x == nx / 2) ds->rho_center = rho;
            if (y == 0 && x == 0) ds->rho_corner = rho;
        }
        if (mode & OBS_SNAP_CMP) acc.change(vx - C(sv.x), vy - C(sv.y));
        if (mode & OBS_SNAP_STORE) vsnap[o] = make_vsnap(vx, vy);
    }
};

// Quantities of a partial in the order of its fields: sums of the mass and of
// rows ny/2 and 0, maxima of |v|, |v - v_snap|, rho and -rho.
constexpr int kObsQ = 7, kObsSums = 3;
static_assert(offsetof(Partial, status) == kObsQ * sizeof(double), "a partial starts with its quantities");

// Quantity `lane` over the warps' values in red, in the warps' order.
template <int NW>
__device__ __forceinline__ double fold_warps(const double* red, int lane, double first)
{
    double x[NW];
#pragma unroll
    for (int w = 0; w < NW; ++w) x[w] = red[min(lane, kObsQ - 1) * NW + w];
    double r = first, m = -1e300;
    if (lane < kObsSums) {
#pragma unroll
        for (int w = 0; w < NW; ++w) r += x[w];
        return r;
    }
#pragma unroll
    for (int w = 0; w < NW; ++w) m = fmax(m, x[w]);
    return m;
}

// The CTA's partial from its threads' reductions (warp shuffles, then the
// warps in order), and in the last CTA to get here the fold of all partials.
// One lane of the first warp takes each quantity, so that the serial chain is
// one FP64 operation a warp and not seven: FP64 operations take 64 cycles
// here, and a CTA's whole reduction is as long as several rows of its walk.
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
    // (few warps hold part of a probe row)
    if (__any_sync(0xffffffffu, acc.row_mid != 0.0)) acc.row_mid = warp_sum(acc.row_mid);
    if (__any_sync(0xffffffffu, acc.row0 != 0.0)) acc.row0 = warp_sum(acc.row0);
    const double v[kObsQ] = {warp_sum(acc.dmass), acc.row_mid, acc.row0,
                             double(warp_max(acc.mv2 != acc.mv2 ? obs_huge<C>() : acc.mv2)),      // |v|^2 (NaN -> huge)
                             double(warp_max(acc.mdv2 != acc.mdv2 ? obs_huge<C>() : acc.mdv2)),
                             double(warp_max(acc.dmax)), double(warp_max(acc.ndmin))};
    const unsigned wbad = __reduce_or_sync(0xffffffffu, bad);
    if (lane == 0) {
#pragma unroll
        for (int j = 0; j < kObsQ; ++j) red[j * NW + wid] = v[j];
        sbad[wid] = wbad;
    }
    __syncthreads();
    const unsigned nparts = gridDim.x * gridDim.y;
    if (wid == 0) {
        const double ref = double(k.rho_ref);
        double r = fold_warps<NW>(red, lane, lane == 0 ? cta_nodes * ref : 0.0);
        const unsigned pb = __reduce_or_sync(0xffffffffu, lane < NW ? sbad[lane] : 0u);
        // roots and densities of the maxima: both are monotone, so of the CTA's as of each warp's
        if (lane == 3 || lane == 4) r = double(sqrt(C(r)));
        else if (lane == 5) r = ref + r;
        else if (lane == 6) r = -(ref - r);
        Partial* p = parts + (blockIdx.y * gridDim.x + blockIdx.x);
        if (lane < kObsQ) reinterpret_cast<double*>(p)[lane] = r;
        else if (lane == kObsQ) p->status = pb;
        __threadfence();
        __syncwarp();
        if (lane == 0) *last = atomicAdd(ticket, 1u) == nparts - 1;
    }
    __syncthreads();
    if (!*last) return;

    // The last CTA: every partial is written and fenced.  A warp folds each
    // quantity in a fixed order (lane l takes partials l, l + 32, ..., then
    // shuffles), so the three sums run on FP64 pipes of their own.
    __threadfence();
    for (int q = wid; q <= kObsQ; q += NW) {
        if (q == kObsQ) {   // the status words
            unsigned b = 0;
            for (unsigned i = lane; i < nparts; i += 32) b |= __ldcg(&parts[i].status);
            b = __reduce_or_sync(0xffffffffu, b);
            if (lane == 0) ds->status = b | (status ? *status : 0u);
            continue;
        }
        const double* x = reinterpret_cast<const double*>(parts) + q;
        constexpr size_t stride = sizeof(Partial) / sizeof(double);
        double r = q < kObsSums ? 0.0 : -1e300;
        if (q < kObsSums) {
#pragma unroll 8
            for (unsigned i = lane; i < nparts; i += 32) r += __ldcg(x + i * stride);
            r = warp_sum(r);
        } else {
#pragma unroll 8
            for (unsigned i = lane; i < nparts; i += 32) r = fmax(r, __ldcg(x + i * stride));
            r = warp_max(r);
        }
        if (lane == 0) {
            switch (q) {
            case 0: ds->mass = r; break;
            case 1: ds->rho_row_mid = r / nx; break;
            case 2: ds->rho_row0 = r / nx; break;
            case 3: ds->max_v = r; break;
            case 4: ds->max_dv = r; break;
            case 5: ds->rho_max = r; break;
            case 6: ds->rho_min = -r; break;
            }
        }
    }
    if (threadIdx.x == 0) *ticket = 0;   // ready for the next launch
}

// One CTA per (strip, row chunk), as the step kernel.  Every CTA reaches the
// reduction, whatever happened to its walk (a misaligned buffer, an empty
// chunk, a stage wait that gave up), so the ticket always completes.
template <typename T, typename C, int NT, int NS, int MINB, bool HALO1>
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
        strip_walk<T, C, NT, NS, true, HALO1, true>(fin, nx, ny, x0, y0, y1, (blockIdx.y & 1) != 0, k, sm, G, bad,
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

// The same with the walk of tiles: `items` pieces of the lattice, each a
// 32-column strip's chunk of `rows` rows, shared out over the grid's CTAs, so
// that a CTA reduces once whatever the lattice's shape.  (With a CTA a piece,
// wide flat lattices were mostly reductions: lbm_stats at 65536 x 16 took 105
// us, now 51; 4096 x 256 100, now 51.)  Pieces of more than 56 rows are worth
// a CTA each, which evens out the last wave: FP64, 2047 x 2049 (80 rows) 1555 us
// shared out and 1436 so, 2048 x 2048 (64 rows) 1493 and 1457.
template <typename T, typename C, int CTAS>
__global__ void __launch_bounds__(kWalkThreads, CTAS)
k_observe_walk(const T* __restrict__ fin, int nx, int ny, int rows, unsigned strips, unsigned items, Coef<C> k, int mode,
               VSnap<C>* __restrict__ vsnap, Partial* __restrict__ parts, unsigned* __restrict__ ticket,
               DevStats* __restrict__ ds, const unsigned* __restrict__ status)
{
    constexpr int NW = kWalkThreads / 32;
    __shared__ WalkPsi<C> sm;
    __shared__ double red[7 * NW];
    __shared__ unsigned sbad[NW], last;
    ObsNode<C> node{mode, nx, ny, ds, vsnap, {}};
    unsigned bad = 0;
    double nodes = 0.0;
    for (unsigned it = blockIdx.x; it < items; it += gridDim.x) {
        const RowChunk c = row_chunk(it / strips, rows, ny);
        const int x0 = int(it % strips) * kWalkW, w = min(kWalkW, nx - x0);
        tile_walk<T, C>(fin, nx, ny, x0, w, c.y0, c.y1, k, sm, bad, node);
        nodes += double(c.y1 - c.y0) * double(w);
        __syncthreads();   // psi of this piece is read
    }
    reduce_and_fold<C, kWalkThreads>(node.acc, bad, nodes, k, nx, red, sbad, &last, parts, ticket, ds, status);
}

// The tile [x0, x0 + w) x [y0, y0 + h) as step_tile takes it, each node handed to
// `node` with its pulled populations and the psi stencil around it; every thread
// of the CTA calls it.  (Sharing this with step_tile through a callable made
// the step 1 to 2 % slower on small lattices.)
template <typename T, typename C, class Node>
__device__ __forceinline__ void tile_nodes(const T* __restrict__ fin, int nx, int ny, int x0, int y0, int w, int h,
                                           const Coef<C>& k, C* __restrict__ sp, unsigned& bad, Node node)
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
        const Stencil<C> q{sp[c], sp[c + 1], sp[c + W], sp[c - 1], sp[c - W],
                           sp[c + W + 1], sp[c + W - 1], sp[c - W - 1], sp[c - W + 1]};
        node(y0 + ly, x0 + lx, g, q);
    }
}

// Tile i of sx x sy nearly equal ones, as plan_tiles cuts them.
struct Tile { int x0, y0, w, h; };
__device__ __forceinline__ Tile tile_at(unsigned i, int sx, int sy, int nx, int ny)
{
    const long long tx = i % unsigned(sx), ty = i / unsigned(sx);
    const int x0 = int(tx * nx / sx), y0 = int(ty * ny / sy);
    return Tile{x0, y0, int((tx + 1) * nx / sx) - x0, int((ty + 1) * ny / sy) - y0};
}

// The moment fields alone, on the generic step's tiles: one round of loads a
// CTA, whose other CTAs hide it, and no barrier between tiles.
template <typename T, typename C>
__global__ void __launch_bounds__(kTileThreads)
k_moments_tile(const T* __restrict__ fin, int nx, int ny, int sx, int sy, Coef<C> k, double* __restrict__ rho_o,
               double* __restrict__ vx_o, double* __restrict__ vy_o)
{
    __shared__ C sp[kTilePsi];
    const Tile t = tile_at(blockIdx.x, sx, sy, nx, ny);
    unsigned bad = 0;   // (no status without a reduction)
    tile_nodes<T, C>(fin, nx, ny, t.x0, t.y0, t.w, t.h, k, sp, bad, [&](int y, int x, C (&g)[9], const Stencil<C>& q) {
        C Fx, Fy, d, vx, vy;
        force<C>(q, k, Fx, Fy);
        node_velocity<C>(g, Fx, Fy, k, d, vx, vy);
        const size_t o = (size_t)y * nx + x;
        rho_o[o] = double(k.rho_ref) + double(d);
        vx_o[o] = double(vx);
        vy_o[o] = double(vy);
    });
}

template <typename T, typename C, int NT, int NS, int MINB, bool HALO1>
int launch_strip(const lbm_params* p, const void* f, int mode, double* rho, double* vx, double* vy, void* vsnap,
           Partial* parts, unsigned* ticket, DevStats* ds, const unsigned* status, cudaStream_t s)
{
    constexpr size_t smem = strip_smem<T, C, NT, NS>();
    static_assert(smem >= (7 * sizeof(double) + sizeof(unsigned)) * (NT / 32) + sizeof(unsigned), "reduction scratch");
    auto kern = k_observe_strip<T, C, NT, NS, MINB, HALO1>;
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
int launch_walk(const lbm_params* p, const void* f, int mode, void* vsnap, Partial* parts, unsigned* ticket, DevStats* ds,
                const unsigned* status, int nsm, cudaStream_t s)
{
    const WalkPlan w = plan_walk(p->nx, p->ny, nsm, CTAS);
    const unsigned items = unsigned(w.sx) * unsigned(w.sy);
    const unsigned grid = w.rows > 56 ? items : std::min(items, unsigned(CTAS * nsm));
    k_observe_walk<T, C, CTAS><<<grid, kWalkThreads, 0, s>>>(
        (const T*)f, p->nx, p->ny, w.rows, unsigned(w.sx), items, make_coef<C>(*p), mode, (VSnap<C>*)vsnap, parts, ticket, ds, status);
    return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_E_CUDA;
}

template <typename T, typename C>
int launch_moments(const lbm_params* p, const void* f, double* rho, double* vx, double* vy, int nsm, cudaStream_t s)
{
    const TilePlan t = plan_tiles(p->nx, p->ny, sizeof(C) == sizeof(double), nsm, INT_MAX);
    k_moments_tile<T, C><<<unsigned(t.sx) * unsigned(t.sy), t.threads, 0, s>>>((const T*)f, p->nx, p->ny, t.sx, t.sy,
                                                                              make_coef<C>(*p), rho, vx, vy);
    return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_E_CUDA;
}

}  // namespace

// FP32 from 3 * 2^20 nodes, where strips of 512 columns idle on at most a
// third of their columns (nx % 4 == 0): the strip walk, whose bulk copies keep
// more of a large lattice in flight.  Everything else: walks of tiles, which
// spread over more CTAs and take any width.  lbm_stats, walk of tiles and
// strip walk (three lattices in turn; us): 2048 x 1024 64 and 75, 1536 x 1536
// 76 and 76, 1028 x 2600 77 and 89, 3000 x 1000 79 and 80, 384 x 8192 80 and
// 78, 768 x 4096 80 and 85, 900 x 4096 93 and 85, 2048 x 2048 102 and 86,
// 4096 x 4096 322 and 211; by idle columns at 8192 rows, 1000 columns 189 and
// 125, 768 137 and 123, 640 114 and 124, 560 114 and 124, and 256 x 16384 102
// and 114.  FP64 lattices walk at any size: 1024 x 1024 322 us, 2048 x 2048 1132,
// 4096 x 4096 4242 (strips, before one division a velocity component did, 458,
// 1420 and 5506).  Flat lattices, of one or a few rows and so many columns that
// every walking CTA would take several pieces of mostly idle warps, keep the
// strips: 131072 x 1 30 us and 52 (FP64 125 and 171), 400000 x 3 63 and 88 (FP64
// 697 and 580: only single rows).
// Strips of 512 columns, four CTAs of 128 threads an SM, the left halo's psi
// off the copying warp: 75.8 us at 1536 x 1536 and 212.2 at 4096 x 4096;
// 1024 columns take 89.9 and 224.6, 2048 columns 99.8 and 249.6.
constexpr long long kObsStripNodes = 3 << 20;
// The moment fields alone: the generic step's tiles, but FP32 strips from 2^23
// nodes.  (us, tiles / walk of tiles / strips: 1023 x 1021 33 / 39 / -, 1024 x
// 1024 33 / 39 / 71, 2048 x 2048 84 / 107 / 90, 33 x 4096 20 / 25 / -, 640 x 8192
// 102 / 133 / 134, 4096 x 4096 286 / 351 / 255.  FP64, with two divisions a
// velocity component: 1024 x 1024 316 / 382 / 447, 2048 x 2048 1169 / 1352 / 1418,
// 33 x 4096 74 / 122 / -, 4096 x 4096 4598 / 5305 / 5413; with one, tiles take 250,
// 919, 54 and 3602.)
constexpr long long kMomentStripNodes = 1 << 23;

int observe_launch(const lbm_params* p, const void* f, int mode, double* rho, double* vx, double* vy, void* vsnap,
                   Partial* parts, unsigned* ticket, DevStats* ds, const unsigned* status, int nsm, cudaStream_t s)
{
    const bool fp64 = p->precision == LBM_FP64, strips = lbm_strip_supported(p);
    const long long nodes = (long long)p->nx * p->ny, padded = (p->nx + 511LL) / 512 * 512;
    const bool covered = strips && !fp64 && 2 * padded <= 3LL * p->nx;
    if (!(mode & OBS_REDUCE) && !(covered && nodes >= kMomentStripNodes))   // the moment fields alone
        return fp64 ? launch_moments<double, double>(p, f, rho, vx, vy, nsm, s)
                    : launch_moments<float, float>(p, f, rho, vx, vy, nsm, s);
    const bool flat = strips && p->ny < (fp64 ? 2 : kWalkH) && (p->nx - 1) / kWalkW >= 2 * kWalkCtas * nsm;
    if (flat && fp64)
        return launch_strip<double, double, 64, 4, 2, false>(p, f, mode, rho, vx, vy, vsnap, parts, ticket, ds, status, s);
    if (!fp64 && (flat || (covered && nodes >= kObsStripNodes)))
        return launch_strip<float, float, 128, 2, 4, true>(p, f, mode, rho, vx, vy, vsnap, parts, ticket, ds, status, s);
    if (fp64) return launch_walk<double, double, 2>(p, f, mode, vsnap, parts, ticket, ds, status, nsm, s);
    return launch_walk<float, float, kWalkCtas>(p, f, mode, vsnap, parts, ticket, ds, status, nsm, s);
}

}  // namespace lbm
