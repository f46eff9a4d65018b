// lbm_host.h -- host-side helpers of liblbm shared by its translation units.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "lbm.h"
// LBM_HOST_ARITHMETIC: the per-node arithmetic compiled by a host compiler
// (a test build, with __device__ and __forceinline__ defined beforehand)
#if defined(__CUDACC__) || defined(LBM_HOST_ARITHMETIC)
#include "lbm_device.cuh"
#endif

extern "C" {
double lbm_tc(void);
int lbm_maxwell(double T_over_Tc, double* rho_v, double* rho_l);
}

// LBM_OK or LBM_E_INVALID / LBM_E_UNSUPPORTED for a parameter set.
int lbm_validate_params(const lbm_params* p);

// LBM_OK or LBM_E_INVALID for the arguments of a built-in field (lbm_init_preset).
int lbm_validate_preset(int nx, int ny, int kind, double size, double width, int32_t cell);

// Tiles of the generic step: the lattice cut into sx x sy nearly equal tiles,
// one CTA of `threads` threads each.
struct TilePlan { int sx, sy, threads; };
constexpr int kTileNodes = 256, kTileThreads = 384, kTilePsi = 400;   // limits of a tile: nodes, threads, psi values
TilePlan plan_tiles(int nx, int ny, bool fp64, int nsm, int max_sy = 65535);   // (rows of a 2-D grid)
// Strips of 32 columns and chunks of `rows` rows of the walks of tiles
// (lbm_tilewalk.cuh), one CTA each, `ctas` of which an SM holds.
struct WalkPlan { int sx, sy, rows; };
WalkPlan plan_walk(int nx, int ny, int nsm, int ctas);

// Room for n records in a device table of cap: the larger buffer is allocated
// before the old one is given back, so that a failed allocation (alloc returns
// null; false) leaves the table as it was.
template <typename T, class Alloc, class Free>
bool table_reserve(T*& table, int& cap, size_t n, Alloc alloc, Free release)
{
    if (n <= (size_t)cap) return true;
    void* const p = alloc(n * sizeof(T));
    if (!p) return false;
    if (table) release(table);
    table = static_cast<T*>(p);
    cap = (int)n;
    return true;
}

// Polls of a bounded stage wait (mbarrier try_wait) before the staged kernels
// declare a row copy stuck, flag a timeout, drain and return.
constexpr long long kStageWaitPolls = 1ll << 26;

// Pipelined strip kernel (lbm_strip*.cu): whether it supports p, its tuning
// configurations (threads per CTA, row stages), and one step with one of them.
// first_wait: polls of each CTA's first stage wait (the others make
// kStageWaitPolls); 0 makes that wait give up at once, as a stuck copy would
// (the failure-detection test of the timeout path).
struct StripConfig { int threads, stages, warp; };
bool lbm_strip_supported(const lbm_params* p);
int lbm_strip_config_count(int precision);
StripConfig lbm_strip_config(int precision, int cfg);
int lbm_strip_launch(const lbm_params* p, int cfg, const void* fin, void* fout, unsigned* status, cudaStream_t s,
                     long long first_wait = kStageWaitPolls);

#if defined(__CUDACC__) || defined(LBM_HOST_ARITHMETIC)
// Kernel constants of a parameter set in the compute type C: the FP32 path's
// Coef<float>, or Coef<double>.
template <typename C>
lbm::Coef<C> make_coef(const lbm_params& p)
{
    lbm::Coef<C> k;
    const double li_c = p.forcing == LBM_LI ? p.sigma / (p.tau - 0.5) : 0.0;
    if constexpr (sizeof(C) == sizeof(double)) {
        const double om = 1.0 / p.tau, pre = 1.0 - 0.5 / p.tau;
        k.T = p.T_over_Tc * lbm_tc();
        k.K2 = 2.0 * p.K;
        k.half_A = 0.5 * p.A;
        k.one_m_A = 1.0 - p.A;
        k.omega = om;
        k.one_m_omega = 1.0 - om;
        k.tau = p.tau;
        k.rho_ref = 0.0;
        k.li_c = li_c;
        k.w3 = 3.0 * om;
        k.w45 = 4.5 * om;
        k.g3 = 3.0 * pre;
        k.g9 = 9.0 * pre;
        k.e0 = (1.0 - p.s_e) / 36.0;
        k.e1 = p.s_e / 12.0;
        k.e2 = p.s_e / 18.0;
        k.e3 = (1.0 - 0.5 * p.s_e) / 6.0;
        k.p0 = (1.0 - p.s_eps) / 36.0;
        k.p1 = p.s_eps / 36.0;
        k.p2 = p.s_eps / 12.0;
        k.p3 = (1.0 - 0.5 * p.s_eps) / 6.0;
        k.q0 = (1.0 - p.s_q) / 12.0;
        k.q1 = p.s_q / 12.0;
        k.q2 = (1.0 - 0.5 * p.s_q) / 12.0;
        k.n0 = (1.0 - om) / 4.0;
        k.n1 = om / 4.0;
        k.n2 = pre / 4.0;
        return k;
    } else {
        k.T = C(p.T_over_Tc * lbm_tc());
        k.K = C(p.K);
        k.s_e = C(p.s_e);
        k.s_eps = C(p.s_eps);
        k.s_q = C(p.s_q);
        k.rho_ref = C(p.rho_ref);
        k.li_c = C(li_c);
        // omega and Guo's 1 - omega/2 both exact floats (omega moved by at most
        // one ulp of 1 - omega/2 where needed), so that the momentum a step adds,
        // omega F/2 + (1 - omega/2) F, is exactly F; the Shan-Chen shift
        // tau = 1/omega as hi + lo.
        k.A = C(p.A);
        k.h_e = C(1.0f - 0.5f * float(p.s_e));
        k.h_eps = C(1.0f - 0.5f * float(p.s_eps));
        k.h_q = C(1.0f - 0.5f * float(p.s_q));
        float om = float(1.0 / p.tau);
        float gp = float(1.0 - 0.5 * double(om));
        if (double(gp) != 1.0 - 0.5 * double(om)) om = float(2.0 * (1.0 - double(gp)));
        k.omega = C(om);
        k.guo_pre = C(gp);
        const double t = 1.0 / double(om);
        k.tau = C(t);
        k.tau_lo = C(t - double(k.tau));
        return k;
    }
}
#endif  // __CUDACC__ || LBM_HOST_ARITHMETIC
