// lbm_fields.cuh -- the built-in initial density fields (slab, droplet,
// bubble, droplet array: a tanh interface plus seeded noise; the paper states
// no initial condition) evaluated per node on the device, for single
// lattices and for batched instances.
#pragma once
#include <cuda_runtime.h>

#include "lbm.h"

namespace lbm {

struct PresetField {
    int kind, nx, ny, cell;
    double size, width, rho_l, rho_v, noise_amp;
    unsigned long long seed;
};

__device__ __forceinline__ unsigned long long splitmix64_dev(unsigned long long x)
{
    unsigned long long z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// 4 / width, held finite: below 2e-308 the quotient would be infinite, and a
// node on the interface (distance 0) 0 * inf instead of halfway.
__device__ __forceinline__ double preset_inv_width4(double width) { return fmin(4.0 / width, 1.7976931348623157e308); }

// rho0 of node (x, y) (inv_width4 = preset_inv_width4(width)): rho_v + (rho_l - rho_v) in + noise with
// in = (1 - tanh(2 d / width))/2 and d the signed distance to the liquid (a
// bubble swaps the phases).
//
// Bound by the FP64 pipe, which is 1/60 of the FP32 one here: hypot, two
// divisions and tanh are some 150 FP64 instructions.  So
//   - centres are half-integers, so the squared distance (in units of 1/4) is
//     an integer, and its correctly rounded root replaces hypot;
//   - (1 - tanh z)/2 = 1/(1 + exp(2z)), which also loses nothing to
//     cancellation on the vapour side;
//   - where an FP32 estimate of the distance (good to 1e-6 of the lengths it
//     is made of) puts the node more than ten widths (z = 20) from the
//     interface, in is 0 or 1 to 5e-18, and neither is evaluated.
__device__ __forceinline__ double preset_density(const PresetField& f, double inv_width4, int x, int y)
{
    unsigned long long q = 0;   // (2 distance)^2 to the centre; slab: 2 distance to the mid-row
    if (f.kind == LBM_SLAB) {
        const long long dy = 2ll * y - f.ny;
        q = (unsigned long long)(dy < 0 ? -dy : dy);
    } else {
        long long dx, dy;
        if (f.kind == LBM_DROPLET_ARRAY) {   // the centre of the node's cell
            dx = 2ll * (x % f.cell) - f.cell;
            dy = 2ll * (y % f.cell) - f.cell;
        } else {
            dx = 2ll * x - f.nx;
            dy = 2ll * y - f.ny;
        }
        q = (unsigned long long)(dx * dx) + (unsigned long long)(dy * dy);
    }
    const float r32 = f.kind == LBM_SLAB ? 0.5f * (float)q : 0.5f * sqrtf((float)q);
    const float s32 = (float)f.size;
    const float far = 10.f * (float)f.width + 1e-5f * (r32 + fabsf(s32)) + 1e-6f;
    double in;
    if (r32 - s32 > far) {
        in = 0.0;
    } else if (s32 - r32 > far) {
        in = 1.0;
    } else {
        const double r = f.kind == LBM_SLAB ? 0.5 * (double)q : 0.5 * sqrt((double)q);
        in = 1.0 / (1.0 + exp((r - f.size) * inv_width4));
    }
    double rho = f.kind == LBM_BUBBLE ? f.rho_l + (f.rho_v - f.rho_l) * in : f.rho_v + (f.rho_l - f.rho_v) * in;
    if (f.noise_amp != 0.0) {
        const unsigned long long z = splitmix64_dev(f.seed ^ ((unsigned long long)y * f.nx + x));
        // 2 xi - 1 with xi = (z >> 11) 2^-53, exactly: the integer difference is below 2^53
        const long long t = (long long)(z >> 11) - (1ll << 52);
        rho += f.noise_amp * ((double)t * (1.0 / 4503599627370496.0));
    }
    return rho;
}

}  // namespace lbm
