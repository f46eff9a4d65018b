// lbm_mlp.cu -- the learned warm start's network: a tanh multilayer
// perceptron (inputs T/Tc, tau, A, K, radius -> density profile samples)
// trained and evaluated by hand-written FP32 kernels (forward, backward,
// Adam).  Inputs and outputs are standardised inside the model with affine
// scalings set by the caller.  Parameters are flattened layer by layer as
// [W (out x in, row-major), b], hidden layers first, then the linear output.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "lbm.h"
#include "lbm_async.cuh"

namespace {

constexpr int TS = 16;   // GEMM tile

enum Epi : int { EPI_NONE = 0, EPI_BIAS_TANH = 1, EPI_BIAS = 2, EPI_TANH_BACK = 3 };

// C[m, n] = sum_k A(m, k) B(k, n), A(m, k) = A[m*sam + k*sak], B(k, n) = B[k*sbk + n*sbn],
// with an epilogue: + bias[n] then tanh; + bias[n]; or times (1 - P[m, n]^2)
// (backpropagation through tanh, P the layer output).  Fixed summation order.
template <int EPI>
__global__ void __launch_bounds__(TS * TS)
k_gemm(const float* __restrict__ A, int sam, int sak, const float* __restrict__ B, int sbk, int sbn,
       float* __restrict__ C, int M, int N, int K, const float* __restrict__ bias, const float* __restrict__ P)
{
    __shared__ float sa[TS][TS + 1], sb[TS][TS + 1];
    const int tx = threadIdx.x % TS, ty = threadIdx.x / TS;
    const int m = blockIdx.y * TS + ty, n = blockIdx.x * TS + tx;
    float acc = 0.f;
    for (int k0 = 0; k0 < K; k0 += TS) {
        const int ka = k0 + tx, kb = k0 + ty;
        const int am = blockIdx.y * TS + ty, bn = blockIdx.x * TS + tx;
        sa[ty][tx] = (am < M && ka < K) ? A[(size_t)am * sam + (size_t)ka * sak] : 0.f;
        sb[ty][tx] = (kb < K && bn < N) ? B[(size_t)kb * sbk + (size_t)bn * sbn] : 0.f;
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < TS; ++kk) acc = fmaf(sa[ty][kk], sb[kk][tx], acc);
        __syncthreads();
    }
    if (m < M && n < N) {
        if (EPI == EPI_BIAS_TANH) acc = tanhf(acc + bias[n]);
        else if (EPI == EPI_BIAS) acc = acc + bias[n];
        else if (EPI == EPI_TANH_BACK) { const float p = P[(size_t)m * N + n]; acc *= (1.f - p * p); }
        C[(size_t)m * N + n] = acc;
    }
}

// (x - mean) / std per column.
__global__ void k_standardize(const float* __restrict__ X, float* __restrict__ Y, int n, int d,
                              const float* __restrict__ mean, const float* __restrict__ sd)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n * d) Y[i] = (X[i] - mean[i % d]) / sd[i % d];
}

__global__ void k_destandardize(float* __restrict__ Y, int n, int d, const float* __restrict__ mean,
                                const float* __restrict__ sd)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n * d) Y[i] = Y[i] * sd[i % d] + mean[i % d];
}

// Output delta of the MSE loss in standardised units, d loss / d out =
// 2 (out - t) / (n m), t = (y - mean)/std, and per-row squared error sums.
__global__ void k_loss_delta(const float* __restrict__ out, const float* __restrict__ Y, float* __restrict__ delta,
                             float* __restrict__ row_loss, int n, int m, const float* __restrict__ mean,
                             const float* __restrict__ sd)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    float s = 0.f;
    const float inv = 2.f / (float(n) * float(m));
    for (int j = 0; j < m; ++j) {
        const float t = (Y[(size_t)r * m + j] - mean[j]) / sd[j];
        const float d = out[(size_t)r * m + j] - t;
        delta[(size_t)r * m + j] = inv * d;
        s += d * d;
    }
    row_loss[r] = s;
}

// Column sums of delta (bias gradient), fixed order.
__global__ void k_colsum(const float* __restrict__ delta, float* __restrict__ g, int n, int m)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= m) return;
    float s = 0.f;
    for (int r = 0; r < n; ++r) s += delta[(size_t)r * m + j];
    g[j] = s;
}

// Adam (Kingma & Ba) with bias correction, one parameter.  The contractions of
// its two averages are written out: left to the compiler they differ from
// kernel to kernel, and a network trained by one drifts from the other's by
// 1e-7 of its parameters.
struct Adam { float lr, b1, b2, eps, c1, c2; };
__device__ __forceinline__ void adam_update(float* p, float gi, float* m1, float* m2, const Adam& h)
{
    const float a = fmaf(1.f - h.b1, gi, h.b1 * *m1);
    const float b = fmaf((1.f - h.b2) * gi, gi, h.b2 * *m2);
    *m1 = a;
    *m2 = b;
    *p -= h.lr * (a / h.c1) / (sqrtf(b / h.c2) + h.eps);
}

__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m1,
                       float* __restrict__ m2, int n, Adam h)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) adam_update(p + i, g[i], m1 + i, m2 + i, h);
}

// Rows perm[0..n) of a row-major array.
__global__ void k_gather(const float* __restrict__ src, const int* __restrict__ perm, float* __restrict__ dst, int n, int d)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n * d) dst[i] = src[(size_t)perm[i / d] * d + i % d];
}

// ---------------------------------------------------------------------------
// The network in two launches a minibatch.  A layer at a time it took about
// twenty (standardise, a GEMM per layer and direction, loss, bias sums, Adam,
// two copies), each 3-15 us of latency for a few thousand outputs.  Every sum
// keeps its order (k ascending, one fused multiply-add a term, from zero), so
// predictions, gradients and trained parameters come out bit for bit as from
// the layered kernels.
// 2000 rows in minibatches of 64, two epochs and the final loss: 8.45 ms layer
// by layer, 1.06 ms so (of a minibatch's 15 us k_net takes 9, k_net_grad 2,
// the rest is the two launches); 256 predictions 57 and 34 us with copies.
// ---------------------------------------------------------------------------
constexpr int kMaxLayers = 17;   // 16 hidden layers and the output

struct NetShape {
    int L;                       // layers
    int size[kMaxLayers + 1];    // widths: input, hidden, output
    int w[kMaxLayers], b[kMaxLayers];   // parameter offsets
    int S[kMaxLayers];           // shared-memory row stride of W: a multiple of 4 floats, odd in 16-byte units,
                                 // so that 128-bit reads of one column block by 8 lanes hit all 32 banks
    int sw[kMaxLayers];          // shared-memory offset of W (floats)
    int sb[kMaxLayers];          // the same for its biases
    int wsum;                    // shared-memory floats of all W and biases: the image k_net copies
    int asum, amax;              // padded activation floats of a row, the widest layer's
};
struct NetBufs {
    float* act[kMaxLayers + 1];    // [rows][size]: act[0] the standardised input
    float* delta[kMaxLayers + 1];  // [rows][size]: delta[l] of layer l's output, l >= 1
};
struct NetScale { const float *xm, *xs, *ym, *ys; };
enum : int { NET_PREDICT = 0, NET_LOSS = 1, NET_GRAD = 2 };

__host__ __device__ constexpr int pad4(int n) { return (n + 3) & ~3; }

// Start of a kernel launched before its predecessor has finished.  Such a
// kernel takes no __restrict__ pointers (which would allow loads ahead of the
// wait and through the read-only cache).
__device__ __forceinline__ void pdl_wait_and_release()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// acc[r] += sum_k a[r][k] w[k] in ascending k, one fused multiply-add a term;
// the next 16 terms' reads are under way while these are added.
template <int RPT>
__device__ __forceinline__ void dot_rows(float (&acc)[RPT], const float* __restrict__ w, const float* __restrict__ a,
                                         int P, int n)
{
    float4 wn[4], an[RPT][4];
    auto fetch = [&](int k) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            wn[q] = *reinterpret_cast<const float4*>(w + k + 4 * q);
#pragma unroll
            for (int r = 0; r < RPT; ++r) an[r][q] = *reinterpret_cast<const float4*>(a + r * P + k + 4 * q);
        }
    };
    int k = 0;
    if (n >= 16) fetch(0);
    for (; k + 16 <= n; k += 16) {
        float4 wc[4], ac[RPT][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            wc[q] = wn[q];
#pragma unroll
            for (int r = 0; r < RPT; ++r) ac[r][q] = an[r][q];
        }
        if (k + 32 <= n) fetch(k + 16);
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                acc[r] = fmaf(ac[r][q].x, wc[q].x, acc[r]);
                acc[r] = fmaf(ac[r][q].y, wc[q].y, acc[r]);
                acc[r] = fmaf(ac[r][q].z, wc[q].z, acc[r]);
                acc[r] = fmaf(ac[r][q].w, wc[q].w, acc[r]);
            }
    }
    for (; k < n; ++k)
#pragma unroll
        for (int r = 0; r < RPT; ++r) acc[r] = fmaf(a[r * P + k], w[k], acc[r]);
}
// The same down a column of W: acc[r] += sum_o d[r][o] w[o S].
template <int RPT>
__device__ __forceinline__ void dot_cols(float (&acc)[RPT], const float* __restrict__ w, int S,
                                         const float* __restrict__ d, int P, int n)
{
    float wn[8];
    float4 dn[RPT][2];
    auto fetch = [&](int o) {
#pragma unroll
        for (int q = 0; q < 8; ++q) wn[q] = w[(o + q) * S];
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
            dn[r][0] = *reinterpret_cast<const float4*>(d + r * P + o);
            dn[r][1] = *reinterpret_cast<const float4*>(d + r * P + o + 4);
        }
    };
    int o = 0;
    if (n >= 8) fetch(0);
    for (; o + 8 <= n; o += 8) {
        float wc[8];
        float4 dc[RPT][2];
#pragma unroll
        for (int q = 0; q < 8; ++q) wc[q] = wn[q];
#pragma unroll
        for (int r = 0; r < RPT; ++r) {
            dc[r][0] = dn[r][0];
            dc[r][1] = dn[r][1];
        }
        if (o + 16 <= n) fetch(o + 8);
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                acc[r] = fmaf(dc[r][q].x, wc[4 * q], acc[r]);
                acc[r] = fmaf(dc[r][q].y, wc[4 * q + 1], acc[r]);
                acc[r] = fmaf(dc[r][q].z, wc[4 * q + 2], acc[r]);
                acc[r] = fmaf(dc[r][q].w, wc[4 * q + 3], acc[r]);
            }
    }
    for (; o < n; ++o)
#pragma unroll
        for (int r = 0; r < RPT; ++r) acc[r] = fmaf(d[r * P + o], w[o * S], acc[r]);
}

// All layers for H RPT rows a CTA: forward, and with NET_GRAD the deltas back
// to the first layer.  Weights and biases (175 KB for 5-128-128-128-64) come
// from `image`, which holds them as shared memory wants them: rows padded so
// that both directions read without bank conflicts (forward a lane reads 4 k
// of its output's row, backward consecutive lanes consecutive inputs of one
// row), in a few bulk copies.  A thread keeps RPT rows' sums of one output.
// Bound by latency: the serial sums (128 dependent FMAs a layer, 1 000 cycles
// with their shared-memory reads) and the image's way from L2 to one SM; rows
// are therefore spread over many CTAs.  (Copied out of the parameters row by
// row -- cp.async of 16 bytes or a bulk copy a row -- issuing alone took
// 5 000 to 9 000 cycles.)
template <int H, int RPT, int MODE>
__global__ void __launch_bounds__(256, 1)
k_net(NetShape sh, const float* image, NetScale sc, const float* X, const float* Y, const int* perm, int n, NetBufs buf,
      float* out, float* row_loss, int* timeout)
{
    constexpr int R = H * RPT, NT = 256;
    extern __shared__ __align__(16) float sm[];
    float* const act = sm + sh.wsum;              // [layer][R][pad4(size)]
    float* const dl = act + R * sh.asum;          // two delta rows sets [2][R][amax]
    float* const ty = dl + 2 * R * sh.amax;       // standardised targets [R][m]
    uint64_t* const bar = reinterpret_cast<uint64_t*>(ty + pad4(R * sh.size[sh.L]));
    const int t = threadIdx.x, L = sh.L, r0 = blockIdx.x * R;
    if (t == 0) {
        lbm::mbar_init(bar, 1);
        lbm::fence_mbar_init();
    }
    pdl_wait_and_release();
    if (t == 0) {
        lbm::mbar_arrive_expect_tx(bar, 4u * sh.wsum);
        for (int i = 0; i < sh.wsum; i += 4096) lbm::bulk_g2s(sm + i, image + i, 4u * min(4096, sh.wsum - i), bar);
    }
    // this thread's first input and target: every global read of the row block is under way at once
    const int d0 = sh.size[0], m = sh.size[L];
    const int xr = t / d0, xc = t - xr * d0, yr = t / m, yc = t - yr * m;
    const bool hx = t < R * d0 && r0 + xr < n, hy = MODE != NET_PREDICT && t < R * m && r0 + yr < n;
    const int xrow = hx ? (perm ? perm[r0 + xr] : r0 + xr) : 0, yrow = hy ? (perm ? perm[r0 + yr] : r0 + yr) : 0;
    // (x - mean) / std per column
    const int P0 = pad4(d0);
    auto input = [&](int r, int c, float x, float mean, float sd) {
        const float v = (x - mean) / sd;
        if (MODE == NET_GRAD) buf.act[0][(size_t)(r0 + r) * d0 + c] = v;
        act[r * P0 + c] = v;
    };
    {
        float x = 0.f, xm = 0.f, xs = 1.f, y = 0.f, ym = 0.f, ys = 1.f;
        if (hx) {
            x = X[(size_t)xrow * d0 + xc];
            xm = sc.xm[xc];
            xs = sc.xs[xc];
        }
        if (hy) {
            y = Y[(size_t)yrow * m + yc];
            ym = sc.ym[yc];
            ys = sc.ys[yc];
        }
        if (hx) input(xr, xc, x, xm, xs);
        else if (t < R * d0) act[xr * P0 + xc] = 0.f;
        if (hy) ty[t] = (y - ym) / ys;
    }
    for (int i = t + NT; i < R * d0; i += NT) {   // inputs and targets beyond one a thread
        const int r = i / d0, c = i - r * d0;
        if (r0 + r < n) input(r, c, X[(size_t)(perm ? perm[r0 + r] : r0 + r) * d0 + c], sc.xm[c], sc.xs[c]);
        else act[r * P0 + c] = 0.f;
    }
    if (MODE != NET_PREDICT) {
        for (int i = t + NT; i < R * m; i += NT) {
            const int r = i / m, j = i - r * m;
            if (r0 + r < n) ty[i] = (Y[(size_t)(perm ? perm[r0 + r] : r0 + r) * m + j] - sc.ym[j]) / sc.ys[j];
        }
    }
    __syncthreads();   // the barrier is initialised, inputs and targets are in place
    const bool ok = lbm::mbar_wait(bar, 0);
    if (__syncthreads_or(!ok)) {   // the bounded wait gave up: flag it, wait once more for the copies, stop
        if (t == 0) {
            *timeout = 1;
            lbm::mbar_wait(bar, 0);
        }
        __syncthreads();
        return;
    }
    float* ain = act;
    for (int l = 0; l < L; ++l) {
        const int in = sh.size[l], on = sh.size[l + 1], P = pad4(in), Q = pad4(on);
        float* aout = ain + R * P;
        for (int i = t; i < H * on; i += NT) {
            const int half = H > 1 && i >= on, o = i - half * on;
            const float* W = sm + sh.sw[l] + o * sh.S[l];
            const float* a = ain + half * RPT * P;
            const float bias = sm[sh.sb[l] + o];
            float acc[RPT];
#pragma unroll
            for (int r = 0; r < RPT; ++r) acc[r] = 0.f;
            dot_rows<RPT>(acc, W, a, P, in);
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                const int row = half * RPT + r;
                float v = acc[r] + bias;
                if (l < L - 1) {
                    v = tanhf(v);
                    if (MODE == NET_GRAD && r0 + row < n) buf.act[l + 1][(size_t)(r0 + row) * on + o] = v;
                } else if (MODE == NET_PREDICT && r0 + row < n) {
                    out[(size_t)(r0 + row) * on + o] = v * sc.ys[o] + sc.ym[o];
                }
                aout[row * Q + o] = v;
            }
        }
        __syncthreads();
        ain = aout;
    }
    if (MODE == NET_PREDICT) return;
    // MSE in standardised units: d = out - t, delta = 2 d / (n m), and per row the sum of d^2
    const int Q = pad4(m);
    const float inv = 2.f / (float(n) * float(m));
    for (int i = t; i < R * m; i += NT) {
        const int r = i / m, j = i - r * m;
        float d = 0.f;
        if (r0 + r < n) {
            d = ain[r * Q + j] - ty[i];
            if (MODE == NET_GRAD) buf.delta[L][(size_t)(r0 + r) * m + j] = inv * d;
        }
        if (MODE == NET_GRAD) dl[r * sh.amax + j] = inv * d;
        ain[r * Q + j] = d;
    }
    __syncthreads();
    if (row_loss && t < R && r0 + t < n) {
        float s = 0.f;
        for (int j = 0; j < m; ++j) s += ain[t * Q + j] * ain[t * Q + j];
        row_loss[r0 + t] = s;
    }
    if (MODE != NET_GRAD) return;
    // delta_prev[b, i] = (sum_o delta[b, o] W[o, i]) (1 - act[b, i]^2)
    const float* dcur = dl;
    float* dnext = dl + R * sh.amax;
    float* a = ain;   // activations of layer l's input, found walking back
    for (int l = L - 1; l > 0; --l) {
        const int in = sh.size[l], on = sh.size[l + 1], P = pad4(in), S = sh.S[l];
        a -= R * P;
        const float* W = sm + sh.sw[l];
        for (int i = t; i < H * in; i += NT) {
            const int half = H > 1 && i >= in, c = i - half * in;
            const float* d = dcur + half * RPT * sh.amax;
            float acc[RPT];
#pragma unroll
            for (int r = 0; r < RPT; ++r) acc[r] = 0.f;
            dot_cols<RPT>(acc, W + c, S, d, sh.amax, on);
#pragma unroll
            for (int r = 0; r < RPT; ++r) {
                const int row = half * RPT + r;
                const float p = a[row * P + c];
                const float v = acc[r] * (1.f - p * p);
                dnext[row * sh.amax + c] = v;
                if (r0 + row < n) buf.delta[l][(size_t)(r0 + row) * in + c] = v;
            }
        }
        __syncthreads();
        const float* tmp = dcur;
        dcur = dnext;
        dnext = const_cast<float*>(tmp);
    }
}

// Parameter gradients over n rows, gW[o, i] = sum_b delta[b, o] act[b, i] and
// gb[o] = sum_b delta[b, o] (b ascending), one thread a weight in 16 x 16
// tiles of every layer at once; ADAM: the update applied in place of storing
// them.
template <bool ADAM>
__global__ void __launch_bounds__(256)
k_net_grad(NetShape sh, NetBufs buf, int n, float* params, float* image, float* grads, float* m1, float* m2, Adam h)
{
    __shared__ float sd[64][TS], sa[64][TS];
    int l = 0, tile = blockIdx.x, ti = 0;
    for (;; ++l) {   // the layer this tile belongs to
        ti = (sh.size[l] + TS - 1) / TS;
        const int nt = ti * ((sh.size[l + 1] + TS - 1) / TS);
        if (tile < nt) break;
        tile -= nt;
    }
    const int in = sh.size[l], on = sh.size[l + 1];
    const int o0 = (tile / ti) * TS, i0 = (tile % ti) * TS;
    const int t = threadIdx.x, tx = t % TS, ty = t / TS;
    const int o = o0 + ty, i = i0 + tx;
    const bool wt = o < on && i < in, bias = o < on && i0 == 0 && tx == 0;
    const int at = sh.w[l] + o * in + i, bt = sh.b[l] + o;
    pdl_wait_and_release();
    // the parameters' Adam state is fetched under the sums
    float p = 0.f, u = 0.f, v = 0.f;
    if (ADAM && wt) {
        p = params[at];
        u = m1[at];
        v = m2[at];
    }
    float acc = 0.f, bsum = 0.f;
    for (int b0 = 0; b0 < n; b0 += 64) {
        const int nb = min(64, n - b0);
        float rd[4], ra[4];   // all eight reads in flight together
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int q = ty + TS * j;
            rd[j] = q < nb && o0 + tx < on ? buf.delta[l + 1][(size_t)(b0 + q) * on + o0 + tx] : 0.f;
            ra[j] = q < nb && i < in ? buf.act[l][(size_t)(b0 + q) * in + i] : 0.f;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            sd[ty + TS * j][tx] = rd[j];
            sa[ty + TS * j][tx] = ra[j];
        }
        __syncthreads();
        if (nb == 64) {
#pragma unroll 16
            for (int q = 0; q < 64; ++q) {
                acc = fmaf(sd[q][ty], sa[q][tx], acc);
                bsum += sd[q][ty];
            }
        } else {
            for (int q = 0; q < nb; ++q) {
                acc = fmaf(sd[q][ty], sa[q][tx], acc);
                bsum += sd[q][ty];
            }
        }
        __syncthreads();
    }
    if (wt) {
        if (ADAM) {
            adam_update(&p, acc, &u, &v, h);
            params[at] = p;
            image[sh.sw[l] + o * sh.S[l] + i] = p;
            m1[at] = u;
            m2[at] = v;
        } else {
            grads[at] = acc;
        }
    }
    if (bias) {
        if (ADAM) {
            adam_update(params + bt, bsum, m1 + bt, m2 + bt, h);
            image[sh.sb[l] + o] = params[bt];
        } else {
            grads[bt] = bsum;
        }
    }
}

// The image of the parameters (padding zero).
__global__ void k_net_image(NetShape sh, const float* __restrict__ params, float* __restrict__ image)
{
    for (int l = 0; l < sh.L; ++l) {
        const int in = sh.size[l], on = sh.size[l + 1], S = sh.S[l];
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < on * S; i += gridDim.x * blockDim.x) {
            const int o = i / S, c = i - o * S;
            image[sh.sw[l] + i] = c < in ? params[sh.w[l] + o * in + c] : 0.f;
        }
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < pad4(on); i += gridDim.x * blockDim.x)
            image[sh.sb[l] + i] = i < on ? params[sh.b[l] + i] : 0.f;
    }
}

uint64_t splitmix(uint64_t x)
{
    uint64_t z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

}  // namespace

struct lbm_ws {
    std::vector<int> sizes;          // n_in, hidden..., n_out
    std::vector<size_t> woff, boff;  // parameter offsets per layer
    size_t np = 0;
    float *params = nullptr, *grads = nullptr, *m1 = nullptr, *m2 = nullptr;
    float *xm = nullptr, *xs = nullptr, *ym = nullptr, *ys = nullptr;   // device scalings
    long long t = 0;                 // Adam steps taken
    cudaStream_t stream = nullptr;
    int nsm = 1;                     // SMs of the device
    // per-batch buffers
    int cap = 0;
    std::vector<float*> acts;        // [L+1] activations (acts[0] = standardised input)
    std::vector<float*> deltas;      // [L+1] deltas of the layers' outputs (deltas[0] unused)
    float *rowloss = nullptr, *X = nullptr, *Y = nullptr;
    // training set: rows, targets and two epochs' orders, kept between calls
    // (a program trains in chunks) and released with the network
    int tcap = 0;
    float *tX = nullptr, *tY = nullptr;
    int *perm[2] = {nullptr, nullptr}, *hperm[2] = {nullptr, nullptr};   // device, pinned host
    cudaEvent_t perm_read[2] = {nullptr, nullptr};                       // the copy of hperm[k] is done
    int* timeout = nullptr;          // pinned host flag a kernel sets when its weight copies did not land
    bool fused = false;              // the weights fit in shared memory: k_net and k_net_grad
    NetShape shape;
    float* image = nullptr;          // fused: weights and biases in k_net's shared-memory layout, kept with params
};

namespace {

int ok(cudaError_t e)
{
    if (e == cudaSuccess) return LBM_OK;
    std::fprintf(stderr, "liblbm (mlp): CUDA error %s\n", cudaGetErrorString(e));
    return LBM_E_CUDA;
}
#define W_CUDA(call)                  \
    do {                              \
        int s_ = ok(call);            \
        if (s_ != LBM_OK) return s_;  \
    } while (0)

int nlayers(const lbm_ws* w) { return (int)w->sizes.size() - 1; }
template <typename T>
void release(T*& p)
{
    cudaFree(p);
    p = nullptr;
}

int ensure(lbm_ws* w, int n)
{
    if (n <= w->cap) return LBM_OK;
    w->cap = 0;
    for (float*& p : w->acts) release(p);
    for (float*& p : w->deltas) release(p);
    release(w->rowloss);
    release(w->X);
    release(w->Y);
    w->acts.assign(nlayers(w) + 1, nullptr);
    w->deltas.assign(nlayers(w) + 1, nullptr);
    for (int l = 0; l <= nlayers(w); ++l) W_CUDA(cudaMalloc(&w->acts[l], sizeof(float) * n * w->sizes[l]));
    for (int l = 1; l <= nlayers(w); ++l) W_CUDA(cudaMalloc(&w->deltas[l], sizeof(float) * n * w->sizes[l]));
    W_CUDA(cudaMalloc(&w->rowloss, sizeof(float) * n));
    W_CUDA(cudaMalloc(&w->X, sizeof(float) * n * w->sizes.front()));
    W_CUDA(cudaMalloc(&w->Y, sizeof(float) * n * w->sizes.back()));
    w->cap = n;
    return LBM_OK;
}

// Buffers of a training set of n rows.
int ensure_train(lbm_ws* w, int n)
{
    if (n <= w->tcap) return LBM_OK;
    w->tcap = 0;
    release(w->tX);
    release(w->tY);
    W_CUDA(cudaMalloc(&w->tX, sizeof(float) * n * w->sizes.front()));
    W_CUDA(cudaMalloc(&w->tY, sizeof(float) * n * w->sizes.back()));
    for (int k = 0; k < 2; ++k) {
        release(w->perm[k]);
        if (w->hperm[k]) cudaFreeHost(w->hperm[k]);
        w->hperm[k] = nullptr;
        W_CUDA(cudaMalloc(&w->perm[k], sizeof(int) * n));
        W_CUDA(cudaMallocHost(&w->hperm[k], sizeof(int) * n));
        if (!w->perm_read[k]) W_CUDA(cudaEventCreateWithFlags(&w->perm_read[k], cudaEventDisableTiming));
    }
    w->tcap = n;
    return LBM_OK;
}

// Shared memory of k_net for R rows a CTA.
size_t net_smem(const NetShape& s, int R)
{
    return sizeof(float) * (s.wsum + (size_t)R * (s.asum + 2 * s.amax) + pad4(R * s.size[s.L])) + sizeof(uint64_t);
}

// Shape of the fused kernels; false if the weights and the widest row block
// (8 rows) exceed the shared memory of an SM.
bool make_shape(const lbm_ws* w, NetShape& s)
{
    std::memset(&s, 0, sizeof(s));
    s.L = nlayers(w);
    size_t wsum = 0, asum = 0, amax = 0;
    for (int l = 0; l <= s.L; ++l) {
        s.size[l] = w->sizes[l];
        asum += pad4(w->sizes[l]);
        amax = std::max<size_t>(amax, pad4(w->sizes[l]));
        if (w->sizes[l] > 4096) return false;
    }
    for (int l = 0; l < s.L; ++l) {
        s.w[l] = (int)w->woff[l];
        s.b[l] = (int)w->boff[l];
        s.S[l] = pad4(w->sizes[l]);
        if ((s.S[l] / 4) % 2 == 0) s.S[l] += 4;
        s.sw[l] = (int)wsum;
        wsum += (size_t)s.S[l] * w->sizes[l + 1];
        s.sb[l] = (int)wsum;
        wsum += pad4(w->sizes[l + 1]);
        if (wsum > 60000) return false;
    }
    s.wsum = (int)wsum;
    s.asum = (int)asum;
    s.amax = (int)amax;
    return net_smem(s, 8) <= 227 * 1024;
}

// The image after params were set.
int refresh_image(lbm_ws* w)
{
    if (!w->fused) return LBM_OK;
    k_net_image<<<64, 256, 0, w->stream>>>(w->shape, w->params, w->image);
    return ok(cudaGetLastError());
}

template <int H, int RPT, int MODE>
int launch_net(lbm_ws* w, const float* X, const float* Y, const int* perm, int n, float* out, float* row_loss)
{
    const size_t smem = net_smem(w->shape, H * RPT);
    auto kern = k_net<H, RPT, MODE>;
    static const cudaError_t set = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    W_CUDA(set);
    NetBufs buf;
    std::memset(&buf, 0, sizeof(buf));
    for (int l = 0; l <= w->shape.L; ++l) {
        buf.act[l] = w->acts[l];
        buf.delta[l] = w->deltas[l];
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((n + H * RPT - 1) / (H * RPT));
    lc.blockDim = dim3(256);
    lc.dynamicSmemBytes = smem;
    lc.stream = w->stream;
    lc.attrs = attr;
    lc.numAttrs = 1;
    W_CUDA(cudaLaunchKernelEx(&lc, kern, w->shape, (const float*)w->image, NetScale{w->xm, w->xs, w->ym, w->ys}, X, Y,
                              perm, n, buf, out, row_loss, w->timeout));
    return LBM_OK;
}

// Rows per CTA: two while that leaves no SM a second CTA (a row block costs
// little more than its weight copy, so few rows finish soonest), then four,
// then eight, which share one weight copy.
template <int MODE>
int run_net(lbm_ws* w, const float* X, const float* Y, const int* perm, int n, float* out, float* row_loss)
{
    if (n <= 2 * w->nsm) return launch_net<1, 2, MODE>(w, X, Y, perm, n, out, row_loss);
    if (n <= 4 * w->nsm) return launch_net<1, 4, MODE>(w, X, Y, perm, n, out, row_loss);
    return launch_net<2, 4, MODE>(w, X, Y, perm, n, out, row_loss);
}

template <bool ADAM>
int run_net_grad(lbm_ws* w, int n, const Adam& h)
{
    NetBufs buf;
    std::memset(&buf, 0, sizeof(buf));
    int ntiles = 0;
    for (int l = 0; l <= w->shape.L; ++l) {
        buf.act[l] = w->acts[l];
        buf.delta[l] = w->deltas[l];
        if (l < w->shape.L) ntiles += ((w->sizes[l] + TS - 1) / TS) * ((w->sizes[l + 1] + TS - 1) / TS);
    }
    // the same shared-memory split as k_net: changing it between the two costs an SM drain a launch
    static const cudaError_t set = cudaFuncSetAttribute(k_net_grad<ADAM>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    W_CUDA(set);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(ntiles);
    lc.blockDim = dim3(TS * TS);
    lc.stream = w->stream;
    lc.attrs = attr;
    lc.numAttrs = 1;
    W_CUDA(cudaLaunchKernelEx(&lc, k_net_grad<ADAM>, w->shape, buf, n, w->params, w->image, w->grads, w->m1, w->m2, h));
    return LBM_OK;
}

dim3 tiles(int M, int N) { return dim3((N + TS - 1) / TS, (M + TS - 1) / TS); }

// Forward pass of n rows already in w->X (raw inputs); output (standardised) in acts[L].
int forward(lbm_ws* w, int n)
{
    const int d = w->sizes.front();
    k_standardize<<<(n * d + 255) / 256, 256, 0, w->stream>>>(w->X, w->acts[0], n, d, w->xm, w->xs);
    const int L = nlayers(w);
    for (int l = 0; l < L; ++l) {
        const int in = w->sizes[l], out = w->sizes[l + 1];
        const float* Wl = w->params + w->woff[l];
        const float* bl = w->params + w->boff[l];
        if (l < L - 1)
            k_gemm<EPI_BIAS_TANH><<<tiles(n, out), TS * TS, 0, w->stream>>>(w->acts[l], in, 1, Wl, 1, in, w->acts[l + 1],
                                                                             n, out, in, bl, nullptr);
        else
            k_gemm<EPI_BIAS><<<tiles(n, out), TS * TS, 0, w->stream>>>(w->acts[l], in, 1, Wl, 1, in, w->acts[l + 1], n,
                                                                        out, in, bl, nullptr);
    }
    return ok(cudaGetLastError());
}

// Backward pass for n rows with targets in w->Y: gradient into w->grads, row losses into w->rowloss.
int backward(lbm_ws* w, int n)
{
    const int L = nlayers(w);
    const int m = w->sizes.back();
    k_loss_delta<<<(n + 127) / 128, 128, 0, w->stream>>>(w->acts[L], w->Y, w->deltas[L], w->rowloss, n, m, w->ym, w->ys);
    for (int l = L - 1; l >= 0; --l) {
        const int in = w->sizes[l], out = w->sizes[l + 1];
        const float* delta = w->deltas[l + 1];
        // gW[o, i] = sum_b delta[b, o] acts_l[b, i]
        k_gemm<EPI_NONE><<<tiles(out, in), TS * TS, 0, w->stream>>>(delta, 1, out, w->acts[l], in, 1,
                                                                    w->grads + w->woff[l], out, in, n, nullptr, nullptr);
        k_colsum<<<(out + 127) / 128, 128, 0, w->stream>>>(delta, w->grads + w->boff[l], n, out);
        if (l > 0)   // delta_prev[b, i] = (sum_o delta[b, o] W[o, i]) (1 - acts_l[b, i]^2)
            k_gemm<EPI_TANH_BACK><<<tiles(n, in), TS * TS, 0, w->stream>>>(delta, out, 1, w->params + w->woff[l], in, 1,
                                                                           w->deltas[l], n, in, out, nullptr, w->acts[l]);
    }
    return ok(cudaGetLastError());
}

// LBM_E_TIMEOUT (once) if a kernel before the last synchronisation gave up waiting.
int timed_out(lbm_ws* w)
{
    if (!*w->timeout) return LBM_OK;
    *w->timeout = 0;
    return LBM_E_TIMEOUT;
}

// Loss over n rows X, Y on the device (mean squared error in standardised
// units), and with grad its gradient into w->grads.
int loss_of(lbm_ws* w, const float* X, const float* Y, int n, bool grad, float* loss)
{
    int s = LBM_OK;
    if (w->fused) {
        s = grad ? run_net<NET_GRAD>(w, X, Y, nullptr, n, nullptr, w->rowloss)
                 : run_net<NET_LOSS>(w, X, Y, nullptr, n, nullptr, w->rowloss);
        if (s == LBM_OK && grad) s = run_net_grad<false>(w, n, Adam{});
    } else {
        if (X != w->X) W_CUDA(cudaMemcpyAsync(w->X, X, sizeof(float) * n * w->sizes.front(), cudaMemcpyDeviceToDevice, w->stream));
        if (Y != w->Y) W_CUDA(cudaMemcpyAsync(w->Y, Y, sizeof(float) * n * w->sizes.back(), cudaMemcpyDeviceToDevice, w->stream));
        if ((s = forward(w, n)) == LBM_OK) s = backward(w, n);
    }
    if (s != LBM_OK) return s;
    std::vector<float> rl(n);
    W_CUDA(cudaMemcpyAsync(rl.data(), w->rowloss, sizeof(float) * n, cudaMemcpyDeviceToHost, w->stream));
    W_CUDA(cudaStreamSynchronize(w->stream));
    if ((s = timed_out(w)) != LBM_OK) return s;
    double tot = 0;
    for (float v : rl) tot += v;
    if (loss) *loss = float(tot / (double(n) * w->sizes.back()));
    return LBM_OK;
}

}  // namespace

extern "C" {

int lbm_ws_create(const lbm_ws_cfg* cfg, lbm_ws** out)
{
    if (!cfg || !out || cfg->n_in < 1 || cfg->n_out < 1 || cfg->n_hidden < 1 || cfg->hidden_layers < 1 ||
        cfg->hidden_layers > 16)
        return LBM_E_INVALID;
    *out = nullptr;
    lbm_ws* w = new (std::nothrow) lbm_ws();
    if (!w) return LBM_E_INVALID;
    w->sizes.push_back(cfg->n_in);
    for (int i = 0; i < cfg->hidden_layers; ++i) w->sizes.push_back(cfg->n_hidden);
    w->sizes.push_back(cfg->n_out);
    size_t p = 0;
    for (int l = 0; l < nlayers(w); ++l) {
        w->woff.push_back(p);
        p += (size_t)w->sizes[l + 1] * w->sizes[l];
        w->boff.push_back(p);
        p += w->sizes[l + 1];
    }
    w->np = p;
    w->fused = make_shape(w, w->shape);
    // Glorot-uniform weights from SplitMix64(seed, index), zero biases.
    std::vector<float> h(p, 0.f);
    for (int l = 0; l < nlayers(w); ++l) {
        const double lim = std::sqrt(6.0 / (w->sizes[l] + w->sizes[l + 1]));
        for (size_t i = 0; i < (size_t)w->sizes[l + 1] * w->sizes[l]; ++i) {
            const double xi = double(splitmix(cfg->seed ^ (w->woff[l] + i)) >> 11) * (1.0 / 9007199254740992.0);
            h[w->woff[l] + i] = float(lim * (2.0 * xi - 1.0));
        }
    }
    std::vector<float> one_in(cfg->n_in, 1.f), zero_in(cfg->n_in, 0.f), one_out(cfg->n_out, 1.f),
        zero_out(cfg->n_out, 0.f);
    cudaError_t e = cudaStreamCreateWithFlags(&w->stream, cudaStreamNonBlocking);
    int dev = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&w->nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaMallocHost(&w->timeout, sizeof(int));
    if (e == cudaSuccess) *w->timeout = 0;
    if (e == cudaSuccess) e = cudaMalloc(&w->params, sizeof(float) * p);
    if (e == cudaSuccess && w->fused) e = cudaMalloc(&w->image, sizeof(float) * w->shape.wsum);
    if (e == cudaSuccess) e = cudaMalloc(&w->grads, sizeof(float) * p);
    if (e == cudaSuccess) e = cudaMalloc(&w->m1, sizeof(float) * p);
    if (e == cudaSuccess) e = cudaMalloc(&w->m2, sizeof(float) * p);
    if (e == cudaSuccess) e = cudaMalloc(&w->xm, sizeof(float) * cfg->n_in);
    if (e == cudaSuccess) e = cudaMalloc(&w->xs, sizeof(float) * cfg->n_in);
    if (e == cudaSuccess) e = cudaMalloc(&w->ym, sizeof(float) * cfg->n_out);
    if (e == cudaSuccess) e = cudaMalloc(&w->ys, sizeof(float) * cfg->n_out);
    if (e == cudaSuccess) e = cudaMemcpyAsync(w->params, h.data(), sizeof(float) * p, cudaMemcpyHostToDevice, w->stream);
    if (e == cudaSuccess && refresh_image(w) != LBM_OK) e = cudaErrorUnknown;
    if (e == cudaSuccess) e = cudaMemsetAsync(w->m1, 0, sizeof(float) * p, w->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(w->m2, 0, sizeof(float) * p, w->stream);
    if (e == cudaSuccess) e = cudaMemcpy(w->xm, zero_in.data(), sizeof(float) * cfg->n_in, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(w->xs, one_in.data(), sizeof(float) * cfg->n_in, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(w->ym, zero_out.data(), sizeof(float) * cfg->n_out, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(w->ys, one_out.data(), sizeof(float) * cfg->n_out, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaStreamSynchronize(w->stream);
    if (e != cudaSuccess) {
        lbm_ws_destroy(w);
        return ok(e);
    }
    *out = w;
    return LBM_OK;
}

void lbm_ws_destroy(lbm_ws* w)
{
    if (!w) return;
    if (w->stream) cudaStreamSynchronize(w->stream);
    for (float* p : {w->params, w->grads, w->m1, w->m2, w->xm, w->xs, w->ym, w->ys, w->rowloss, w->X, w->Y, w->tX, w->tY,
                     w->image})
        cudaFree(p);
    for (float* p : w->acts) cudaFree(p);
    for (float* p : w->deltas) cudaFree(p);
    if (w->timeout) cudaFreeHost(w->timeout);
    for (int k = 0; k < 2; ++k) {
        cudaFree(w->perm[k]);
        if (w->hperm[k]) cudaFreeHost(w->hperm[k]);
        if (w->perm_read[k]) cudaEventDestroy(w->perm_read[k]);
    }
    if (w->stream) cudaStreamDestroy(w->stream);
    delete w;
}

int lbm_ws_num_params(lbm_ws* w, int64_t* n)
{
    if (!w || !n) return LBM_E_INVALID;
    *n = (int64_t)w->np;
    return LBM_OK;
}

int lbm_ws_set_scaling(lbm_ws* w, const float* x_mean, const float* x_std, const float* y_mean, const float* y_std)
{
    if (!w || !x_mean || !x_std || !y_mean || !y_std) return LBM_E_INVALID;
    const int d = w->sizes.front(), m = w->sizes.back();
    for (int i = 0; i < d; ++i)
        if (!(x_std[i] > 0)) return LBM_E_INVALID;
    for (int i = 0; i < m; ++i)
        if (!(y_std[i] > 0)) return LBM_E_INVALID;
    W_CUDA(cudaMemcpy(w->xm, x_mean, sizeof(float) * d, cudaMemcpyHostToDevice));
    W_CUDA(cudaMemcpy(w->xs, x_std, sizeof(float) * d, cudaMemcpyHostToDevice));
    W_CUDA(cudaMemcpy(w->ym, y_mean, sizeof(float) * m, cudaMemcpyHostToDevice));
    W_CUDA(cudaMemcpy(w->ys, y_std, sizeof(float) * m, cudaMemcpyHostToDevice));
    return LBM_OK;
}

int lbm_ws_get_params(lbm_ws* w, float* host)
{
    if (!w || !host) return LBM_E_INVALID;
    W_CUDA(cudaMemcpy(host, w->params, sizeof(float) * w->np, cudaMemcpyDeviceToHost));
    return LBM_OK;
}

int lbm_ws_set_params(lbm_ws* w, const float* host)
{
    if (!w || !host) return LBM_E_INVALID;
    // on the network's own stream: a later call's kernels follow the resets
    W_CUDA(cudaMemsetAsync(w->m1, 0, sizeof(float) * w->np, w->stream));
    W_CUDA(cudaMemsetAsync(w->m2, 0, sizeof(float) * w->np, w->stream));
    W_CUDA(cudaMemcpyAsync(w->params, host, sizeof(float) * w->np, cudaMemcpyHostToDevice, w->stream));
    const int s = refresh_image(w);
    if (s != LBM_OK) return s;
    W_CUDA(cudaStreamSynchronize(w->stream));
    w->t = 0;
    return LBM_OK;
}

int lbm_ws_loss_grad(lbm_ws* w, const float* X_host, const float* Y_host, int n, float* loss, float* grad_host)
{
    if (!w || !X_host || !Y_host || n < 1) return LBM_E_INVALID;
    int s = ensure(w, n);
    if (s != LBM_OK) return s;
    W_CUDA(cudaMemcpyAsync(w->X, X_host, sizeof(float) * n * w->sizes.front(), cudaMemcpyHostToDevice, w->stream));
    W_CUDA(cudaMemcpyAsync(w->Y, Y_host, sizeof(float) * n * w->sizes.back(), cudaMemcpyHostToDevice, w->stream));
    if ((s = loss_of(w, w->X, w->Y, n, grad_host != nullptr, loss)) != LBM_OK) return s;
    if (grad_host) {
        W_CUDA(cudaMemcpyAsync(grad_host, w->grads, sizeof(float) * w->np, cudaMemcpyDeviceToHost, w->stream));
        W_CUDA(cudaStreamSynchronize(w->stream));
    }
    return LBM_OK;
}

int lbm_ws_train(lbm_ws* w, const float* X_host, const float* Y_host, int n, int epochs, int batch, float lr,
                 uint64_t seed, float* final_loss)
{
    if (!w || !X_host || !Y_host || n < 1 || epochs < 0 || batch < 1 || !(lr > 0)) return LBM_E_INVALID;
    const int d = w->sizes.front(), m = w->sizes.back();
    batch = batch > n ? n : batch;
    int s = ensure(w, final_loss ? n : batch);
    if (s == LBM_OK) s = ensure_train(w, n);
    if (s != LBM_OK) return s;
    W_CUDA(cudaMemcpyAsync(w->tX, X_host, sizeof(float) * n * d, cudaMemcpyHostToDevice, w->stream));
    W_CUDA(cudaMemcpyAsync(w->tY, Y_host, sizeof(float) * n * m, cudaMemcpyHostToDevice, w->stream));
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    for (int ep = 0; ep < epochs && s == LBM_OK; ++ep) {
        // deterministic per-epoch shuffle (Fisher-Yates on SplitMix64 draws), made on the host while the
        // GPU trains on the epoch before; the rows stay in place and are read through it
        const int k = ep & 1;
        int* perm = w->hperm[k];
        if (ep >= 2 && (s = ok(cudaEventSynchronize(w->perm_read[k]))) != LBM_OK) break;
        for (int i = 0; i < n; ++i) perm[i] = i;
        for (int i = n - 1; i > 0; --i) {
            const int j = int(splitmix(seed ^ ((uint64_t)ep << 32) ^ (uint64_t)i) % (uint64_t)(i + 1));
            const int t = perm[i];
            perm[i] = perm[j];
            perm[j] = t;
        }
        if ((s = ok(cudaMemcpyAsync(w->perm[k], perm, sizeof(int) * n, cudaMemcpyHostToDevice, w->stream))) != LBM_OK) break;
        if ((s = ok(cudaEventRecord(w->perm_read[k], w->stream))) != LBM_OK) break;
        for (int b0 = 0; b0 < n && s == LBM_OK; b0 += batch) {
            const int nb = (n - b0 < batch) ? n - b0 : batch;
            ++w->t;
            const Adam h{lr, b1, b2, eps, 1.f - std::pow(b1, float(w->t)), 1.f - std::pow(b2, float(w->t))};
            if (w->fused) {
                s = run_net<NET_GRAD>(w, w->tX, w->tY, w->perm[k] + b0, nb, nullptr, nullptr);
                if (s == LBM_OK) s = run_net_grad<true>(w, nb, h);
                continue;
            }
            k_gather<<<(nb * d + 255) / 256, 256, 0, w->stream>>>(w->tX, w->perm[k] + b0, w->X, nb, d);
            k_gather<<<(nb * m + 255) / 256, 256, 0, w->stream>>>(w->tY, w->perm[k] + b0, w->Y, nb, m);
            if ((s = forward(w, nb)) != LBM_OK) break;
            if ((s = backward(w, nb)) != LBM_OK) break;
            k_adam<<<(int(w->np) + 255) / 256, 256, 0, w->stream>>>(w->params, w->grads, w->m1, w->m2, int(w->np), h);
            s = ok(cudaGetLastError());
        }
    }
    const int e = ok(cudaStreamSynchronize(w->stream));
    if (s == LBM_OK) s = e;
    if (s == LBM_OK) s = timed_out(w);
    if (s == LBM_OK && final_loss)   // loss over the whole training set with the final parameters
        s = loss_of(w, w->tX, w->tY, n, false, final_loss);
    return s;
}

int lbm_ws_predict(lbm_ws* w, const float* X_host, int n, float* Y_host)
{
    if (!w || !X_host || !Y_host || n < 1) return LBM_E_INVALID;
    int s = ensure(w, n);
    if (s != LBM_OK) return s;
    const int d = w->sizes.front(), m = w->sizes.back();
    W_CUDA(cudaMemcpyAsync(w->X, X_host, sizeof(float) * n * d, cudaMemcpyHostToDevice, w->stream));
    float* outp = w->acts[nlayers(w)];
    if (w->fused) {
        if ((s = run_net<NET_PREDICT>(w, w->X, nullptr, nullptr, n, outp, nullptr)) != LBM_OK) return s;
    } else {
        if ((s = forward(w, n)) != LBM_OK) return s;
        k_destandardize<<<(n * m + 255) / 256, 256, 0, w->stream>>>(outp, n, m, w->ym, w->ys);
        W_CUDA(cudaGetLastError());
    }
    W_CUDA(cudaMemcpyAsync(Y_host, outp, sizeof(float) * n * m, cudaMemcpyDeviceToHost, w->stream));
    W_CUDA(cudaStreamSynchronize(w->stream));
    return timed_out(w);
}

}  // extern "C"
