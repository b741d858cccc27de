/*
 * lb_mlp.cu -- learned interface placement.
 *
 * Sec. 2.2 leaves the switching criterion open (it lists local Knudsen numbers and the
 * B parameter from the literature). This file adds a small network that predicts, per
 * node, whether the high-order set is needed:
 *   features (8, from the node's own populations): Pi^neq_xx / rho, Pi^neq_xy / rho,
 *     Pi^neq_yy / rho, q_x / rho, q_y / rho, wall distance / H, local Kn (Eq. (KN)),
 *     gradient-length Knudsen number Kn |grad rho| / rho;
 *   label (for training): 1 when more than a threshold of the node's non-equilibrium
 *     part lies beyond what a second-order Hermite expansion carries (what a low-order
 *     node can hold, Sec. 2.2), measured on a high-order run;
 *   network: 8 -> 64 -> 64 -> 1, GELU (erf form) hidden layers, sigmoid output.
 * Training runs here in FP32 (mini-batch training in one cluster kernel; whole-set gradients
 * as a forward, a backward, a weight-gradient and an Adam kernel each);
 * inference uses BF16 weights with FP32 accumulation. Parameter layout:
 * W1 [64][8], b1 [64], W2 [64][64], b2 [64], W3 [64], b3 [1] (4801 values).
 */
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "../../include/lb.h"
#include "lb_mlp.h"

namespace lbm {

constexpr int NF = 8, NH = 64;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + NH * NF, OFF_W2 = OFF_B1 + NH, OFF_B2 = OFF_W2 + NH * NH,
              OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NH, NPARAM = OFF_B3 + 1;
static_assert(NPARAM == 4801, "parameter count");

__device__ __forceinline__ float gelu(float a) { return 0.5f * a * (1.0f + erff(a * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float a)
{
    return 0.5f * (1.0f + erff(a * 0.70710678118654752f)) + a * expf(-0.5f * a * a) * 0.39894228040143268f;
}

/* Forward pass of samples 0 .. B - 1 (columns of X [NF][n]); keeps the pre-activations and
 * activations for the backward pass. One thread per sample. */
__global__ void fwd_kernel(const float *__restrict__ th, const float *__restrict__ norm, const float *__restrict__ X,
                           long long n, int B, float *xn, float *a1, float *h1, float *a2,
                           float *h2, float *pout)
{
    __shared__ float s[NPARAM];
    for (int k = threadIdx.x; k < NPARAM; k += blockDim.x) s[k] = th[k];
    __syncthreads();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    const long long c = b;
    float x[NF];
    for (int f = 0; f < NF; ++f) {
        x[f] = (X[(long long)f * n + c] - norm[f]) / norm[NF + f];
        xn[(size_t)b * NF + f] = x[f];
    }
    float hh[NH];
    for (int i = 0; i < NH; ++i) {
        float t = s[OFF_B1 + i];
        for (int f = 0; f < NF; ++f) t = fmaf(s[OFF_W1 + i * NF + f], x[f], t);
        a1[(size_t)b * NH + i] = t;
        hh[i] = gelu(t);
        h1[(size_t)b * NH + i] = hh[i];
    }
    float z = s[OFF_B3];
    for (int i = 0; i < NH; ++i) {
        float t = s[OFF_B2 + i];
        for (int k = 0; k < NH; ++k) t = fmaf(s[OFF_W2 + i * NH + k], hh[k], t);
        a2[(size_t)b * NH + i] = t;
        const float g = gelu(t);
        h2[(size_t)b * NH + i] = g;
        z = fmaf(s[OFF_W3 + i], g, z);
    }
    pout[b] = 1.0f / (1.0f + expf(-z));
}

/* Backward pass through the activations: dz = (p - y) / B, then dA2 and dA1 per sample. */
__global__ void bwd_kernel(const float *__restrict__ th, const float *__restrict__ Y, int B,
                           const float *a1, const float *a2, const float *pout, float *dz, float *da1, float *da2,
                           double *loss_acc)
{
    __shared__ float s[NPARAM];
    for (int k = threadIdx.x; k < NPARAM; k += blockDim.x) s[k] = th[k];
    __syncthreads();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    const float y = Y[b], p = pout[b];
    const float g = (p - y) / (float)B;
    dz[b] = g;
    if (loss_acc) {
        const double pc = fmin(fmax((double)p, 1e-30), 1.0 - 1e-7);
        atomicAdd(loss_acc, -((double)y * log(pc) + (1.0 - (double)y) * log(1.0 - pc)) / (double)B);
    }
    float d2[NH];
    for (int i = 0; i < NH; ++i) {
        d2[i] = g * s[OFF_W3 + i] * gelu_grad(a2[(size_t)b * NH + i]);
        da2[(size_t)b * NH + i] = d2[i];
    }
    for (int k = 0; k < NH; ++k) {
        float t = 0.0f;
        for (int i = 0; i < NH; ++i) t = fmaf(d2[i], s[OFF_W2 + i * NH + k], t);
        da1[(size_t)b * NH + k] = t * gelu_grad(a1[(size_t)b * NH + k]);
    }
}

/* Weight gradients, one thread per parameter, summed over the batch in sample order. */
__global__ void wgrad_kernel(int B, const float *xn, const float *h1, const float *h2, const float *dz, const float *da1,
                             const float *da2, float *grad)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= NPARAM) return;
    float t = 0.0f;
    if (k < OFF_B1) {
        const int i = k / NF, f = k % NF;
        for (int b = 0; b < B; ++b) t = fmaf(da1[(size_t)b * NH + i], xn[(size_t)b * NF + f], t);
    } else if (k < OFF_W2) {
        const int i = k - OFF_B1;
        for (int b = 0; b < B; ++b) t += da1[(size_t)b * NH + i];
    } else if (k < OFF_B2) {
        const int i = (k - OFF_W2) / NH, j = (k - OFF_W2) % NH;
        for (int b = 0; b < B; ++b) t = fmaf(da2[(size_t)b * NH + i], h1[(size_t)b * NH + j], t);
    } else if (k < OFF_W3) {
        const int i = k - OFF_B2;
        for (int b = 0; b < B; ++b) t += da2[(size_t)b * NH + i];
    } else if (k < OFF_B3) {
        const int i = k - OFF_W3;
        for (int b = 0; b < B; ++b) t = fmaf(dz[b], h2[(size_t)b * NH + i], t);
    } else {
        for (int b = 0; b < B; ++b) t += dz[b];
    }
    grad[k] = t;
}

/* Adam (Kingma & Ba), bias-corrected, step t >= 1. */
__global__ void adam_kernel(float *th, float *m, float *v, const float *g, int t, float lr, float b1, float b2, float eps)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= NPARAM) return;
    const float mk = b1 * m[k] + (1.0f - b1) * g[k];
    const float vk = b2 * v[k] + (1.0f - b2) * g[k] * g[k];
    m[k] = mk;
    v[k] = vk;
    const float mh = mk / (1.0f - powf(b1, (float)t)), vh = vk / (1.0f - powf(b2, (float)t));
    th[k] -= lr * mh / (sqrtf(vh) + eps);
}

/* ---- mini-batch training: one thread-block cluster takes every batch of a launch ----
 *
 * A batch of a few hundred samples is about 3.5 M multiply-adds, and the next batch needs
 * the updated weights: the work is a chain of small steps, bound by latency, not by the
 * chip's rate. One launch per layer and batch cost 113 us a batch (a weight gradient that
 * walked the samples one by one in each thread, and five launches). Here a cluster of
 * TR_NC blocks keeps the weights, the activations and Adam's moments on chip for all the
 * batches of a launch: block r takes the batch's samples r B / TR_NC .. in tiles of TR_S,
 * every block writes its gradient sums to its shared memory, and after a cluster barrier
 * block r adds the TR_NC sums of its slice of the parameters in rank order through
 * distributed shared memory, updates it and stores the new values into every block. Two
 * cluster barriers a batch; sums in a fixed order, so a run repeats bit for bit. The next
 * tile's samples (a gather over the shuffled order) are loaded while this one is computed.
 * Measured: 100 000 samples in batches of 256, one epoch 51.9 ms -> 4.8 ms with
 * a cluster of 8 blocks, 4.0 ms with 16 (of which 1 ms is the host's shuffle). */
constexpr int TR_S = 32, TR_T = 512;
constexpr int TR_LD = NH + 4;   /* activation and W2 rows in shared memory: conflict-free 16-byte reads */
static_assert(TR_T == 16 * TR_S && TR_T == 8 * NH, "thread mapping of the training kernel");

struct TrainSmem {
    float w1[NH][NF + 4], w2[NH][TR_LD], b1[NH], b2[NH], w3[NH], b3, pad[3];
    float x[TR_S][NF + 4], y[TR_S];
    float h1[TR_S][TR_LD], g1[TR_S][TR_LD], h2[TR_S][TR_LD], d2[TR_S][TR_LD], d1[TR_S][TR_LD];
    float zp[TR_S][2], dz[TR_S];
    float grad[NPARAM + 3];
};

/* parameter k of the packed vector in a block's shared memory */
__device__ __forceinline__ float *train_param(TrainSmem &s, int k)
{
    if (k < OFF_B1) return &s.w1[k / NF][k % NF];
    if (k < OFF_W2) return &s.b1[k - OFF_B1];
    if (k < OFF_B2) return &s.w2[(k - OFF_W2) / NH][(k - OFF_W2) % NH];
    if (k < OFF_W3) return &s.b2[k - OFF_B2];
    if (k < OFF_B3) return &s.w3[k - OFF_W3];
    return &s.b3;
}

/* Batches of `batch` samples (the last may be short) over samples idx[0 .. count): forward,
 * backward, Adam with step numbers t0 + 1, ...; p of sample idx[k] at its batch's weights
 * goes to pall[k] when pall is not NULL. th, m, v are read at the start and written at the
 * end. Launched as one cluster of TR_NC blocks. */
template <int TR_NC>
__global__ void __launch_bounds__(TR_T, 1)
    train_kernel(float *__restrict__ th, float *__restrict__ m, float *__restrict__ v, const float *__restrict__ norm,
                 const float *__restrict__ X, long long n, const float *__restrict__ Y, const int *__restrict__ idx,
                 int count, int batch, int t0, float lr, float *__restrict__ pall)
{
    namespace cg = cooperative_groups;
    constexpr int TR_SL = (NPARAM + TR_NC - 1) / TR_NC;
    static_assert(TR_SL <= 2 * TR_T, "two parameters of the slice per thread");
    cg::cluster_group cl = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char train_smem[];
    TrainSmem &s = *reinterpret_cast<TrainSmem *>(train_smem);
    const int tid = threadIdx.x, rank = (int)cl.block_rank(), lane = tid & 31;
    for (int k = tid; k < NPARAM; k += TR_T) *train_param(s, k) = th[k];
    /* this thread's parameters of the block's slice, with their Adam moments */
    const int k0 = rank * TR_SL + tid, kend = min(NPARAM, (rank + 1) * TR_SL);
    float mk[2] = {0.0f, 0.0f}, vk[2] = {0.0f, 0.0f};
#pragma unroll
    for (int u = 0; u < 2; ++u)
        if (k0 + u * TR_T < kend) {
            mk[u] = m[k0 + u * TR_T];
            vk[u] = v[k0 + u * TR_T];
        }
    /* samples of tile q of this block in the batch at s0: idx[first .. first + cnt) */
    auto tile = [&](int s0, int q, int &first, int &cnt) {
        const int B = min(batch, count - s0), per = (B + TR_NC - 1) / TR_NC;
        const int lo = rank * per + q * TR_S, hi = min(B, (rank + 1) * per);
        cnt = max(0, min(TR_S, hi - lo));
        first = s0 + lo;
    };
    /* one value of a tile per thread: feature tid / TR_S of sample tid % TR_S (normalised), or
     * the label; 0 beyond the tile's samples */
    const int pf = tid / TR_S, ps = tid % TR_S;
    float nmean = 0.0f, nscale = 1.0f;
    if (pf < NF) {
        nmean = norm[pf];
        nscale = norm[NF + pf];
    }
    auto fetch = [&](int s0, int q) -> float {
        int first, cnt;
        tile(s0, q, first, cnt);
        if (pf > NF || ps >= cnt) return 0.0f;
        const long long c = idx[first + ps];
        return pf < NF ? (X[(long long)pf * n + c] - nmean) / nscale : Y[c];
    };
    auto put = [&](float val) {
        if (pf < NF) s.x[ps][pf] = val;
        else if (pf == NF) s.y[ps] = val;
    };
    const int i64 = tid % NH, sg = tid / NH * 4;   /* a unit and four samples */
    const int wi = tid / 16 * 2, wj = tid % 16 * 4;   /* a 2 x 4 block of the W2 gradient */
    put(fetch(0, 0));
    cl.sync();
    int t = t0;
    for (int s0 = 0; s0 < count; s0 += batch) {
        const int B = min(batch, count - s0), nt = ((B + TR_NC - 1) / TR_NC + TR_S - 1) / TR_S;
        float gw2[2][4] = {{0.0f, 0.0f, 0.0f, 0.0f}, {0.0f, 0.0f, 0.0f, 0.0f}}, gw1 = 0.0f, gb = 0.0f;
        for (int q = 0; q < nt; ++q) {
            int first, cnt;
            tile(s0, q, first, cnt);
            const bool last = q + 1 == nt;
            const bool more = !last || s0 + batch < count;
            float nxt = 0.0f;
            if (more) nxt = last ? fetch(s0 + batch, 0) : fetch(s0, q + 1);
            float g2[4], z4[4];
            if (sg < cnt) {   /* layer 1 */
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    float a = s.b1[i64];
#pragma unroll
                    for (int f = 0; f < NF; ++f) a = fmaf(s.w1[i64][f], s.x[sg + u][f], a);
                    const float c = 0.5f * (1.0f + erff(a * 0.70710678118654752f));
                    s.h1[sg + u][i64] = a * c;
                    s.g1[sg + u][i64] = c + a * expf(-0.5f * a * a) * 0.39894228040143268f;
                }
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u) s.h1[sg + u][i64] = 0.0f;
            }
            __syncthreads();
            if (sg < cnt) {   /* layer 2 and the output's dot product */
                float a[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) a[u] = s.b2[i64];
#pragma unroll
                for (int k = 0; k < NH; k += 4) {
                    const float4 w = *reinterpret_cast<const float4 *>(&s.w2[i64][k]);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const float4 h = *reinterpret_cast<const float4 *>(&s.h1[sg + u][k]);
                        a[u] = fmaf(w.x, h.x, a[u]);
                        a[u] = fmaf(w.y, h.y, a[u]);
                        a[u] = fmaf(w.z, h.z, a[u]);
                        a[u] = fmaf(w.w, h.w, a[u]);
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float c = 0.5f * (1.0f + erff(a[u] * 0.70710678118654752f));
                    const float h = a[u] * c;
                    g2[u] = c + a[u] * expf(-0.5f * a[u] * a[u]) * 0.39894228040143268f;
                    s.h2[sg + u][i64] = h;
                    z4[u] = s.w3[i64] * h;
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                    for (int u = 0; u < 4; ++u) z4[u] += __shfl_xor_sync(0xffffffffu, z4[u], o);
                if (lane < 4) s.zp[sg + lane][i64 / 32] = lane == 0 ? z4[0] : (lane == 1 ? z4[1] : (lane == 2 ? z4[2] : z4[3]));
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u) s.h2[sg + u][i64] = 0.0f;
            }
            __syncthreads();
            if (sg < cnt) {   /* dz = (p - y) / B; layer 2's deltas */
                float dzl = 0.0f;
                if (lane < 4) {
                    const int sm = sg + lane;
                    const float p = 1.0f / (1.0f + expf(-(s.b3 + s.zp[sm][0] + s.zp[sm][1])));
                    dzl = sm < cnt ? (p - s.y[sm]) / (float)B : 0.0f;
                    if (i64 < 32) {
                        s.dz[sm] = dzl;
                        if (pall && sm < cnt) pall[first + sm] = p;
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    s.d2[sg + u][i64] = __shfl_sync(0xffffffffu, dzl, u) * s.w3[i64] * g2[u];
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u) s.d2[sg + u][i64] = 0.0f;
                if (i64 < 4) s.dz[sg + i64] = 0.0f;
            }
            __syncthreads();
            if (sg < cnt) {   /* layer 1's deltas */
                float a[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                for (int i = 0; i < NH; i += 4) {
                    const float w0 = s.w2[i][i64], w1 = s.w2[i + 1][i64], w2 = s.w2[i + 2][i64], w3 = s.w2[i + 3][i64];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const float4 d = *reinterpret_cast<const float4 *>(&s.d2[sg + u][i]);
                        a[u] = fmaf(d.x, w0, a[u]);
                        a[u] = fmaf(d.y, w1, a[u]);
                        a[u] = fmaf(d.z, w2, a[u]);
                        a[u] = fmaf(d.w, w3, a[u]);
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) s.d1[sg + u][i64] = a[u] * s.g1[sg + u][i64];
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u) s.d1[sg + u][i64] = 0.0f;
            }
            const int ns = (cnt + 3) & ~3;   /* rows up to here are filled */
            for (int b = 0; b < ns; ++b) {
                const float2 d = *reinterpret_cast<const float2 *>(&s.d2[b][wi]);
                const float4 h = *reinterpret_cast<const float4 *>(&s.h1[b][wj]);
                gw2[0][0] = fmaf(d.x, h.x, gw2[0][0]);
                gw2[0][1] = fmaf(d.x, h.y, gw2[0][1]);
                gw2[0][2] = fmaf(d.x, h.z, gw2[0][2]);
                gw2[0][3] = fmaf(d.x, h.w, gw2[0][3]);
                gw2[1][0] = fmaf(d.y, h.x, gw2[1][0]);
                gw2[1][1] = fmaf(d.y, h.y, gw2[1][1]);
                gw2[1][2] = fmaf(d.y, h.z, gw2[1][2]);
                gw2[1][3] = fmaf(d.y, h.w, gw2[1][3]);
            }
            __syncthreads();
            for (int b = 0; b < ns; ++b) gw1 = fmaf(s.d1[b][tid / NF], s.x[b][tid % NF], gw1);
            if (tid < NH) {
                for (int b = 0; b < ns; ++b) gb += s.d1[b][tid];
            } else if (tid < 2 * NH) {
                for (int b = 0; b < ns; ++b) gb += s.d2[b][tid - NH];
            } else if (tid < 3 * NH) {
                for (int b = 0; b < ns; ++b) gb = fmaf(s.dz[b], s.h2[b][tid - 2 * NH], gb);
            } else if (tid == 3 * NH) {
                for (int b = 0; b < ns; ++b) gb += s.dz[b];
            }
            __syncthreads();
            if (more) put(nxt);
            if (!last) __syncthreads();
        }
        s.grad[OFF_W1 + tid] = gw1;
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) s.grad[OFF_W2 + (wi + a) * NH + wj + b] = gw2[a][b];
        if (tid < NH) s.grad[OFF_B1 + tid] = gb;
        else if (tid < 2 * NH) s.grad[OFF_B2 + tid - NH] = gb;
        else if (tid < 3 * NH) s.grad[OFF_W3 + tid - 2 * NH] = gb;
        else if (tid == 3 * NH) s.grad[OFF_B3] = gb;
        cl.sync();   /* every block's sums are in place */
        t += 1;
        const float c1 = 1.0f - powf(0.9f, (float)t), c2 = 1.0f - powf(0.999f, (float)t);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int k = k0 + u * TR_T;
            if (k >= kend) continue;
            float gr[TR_NC];
#pragma unroll
            for (int r = 0; r < TR_NC; ++r) gr[r] = *cl.map_shared_rank(&s.grad[k], r);
            float g = gr[0];
#pragma unroll
            for (int r = 1; r < TR_NC; ++r) g += gr[r];
            mk[u] = 0.9f * mk[u] + (1.0f - 0.9f) * g;
            vk[u] = 0.999f * vk[u] + (1.0f - 0.999f) * g * g;
            const float nw = *train_param(s, k) - lr * (mk[u] / c1) / (sqrtf(vk[u] / c2) + 1e-8f);
#pragma unroll
            for (int r = 0; r < TR_NC; ++r) *cl.map_shared_rank(train_param(s, k), r) = nw;
        }
        cl.sync();   /* the new weights are in place, the sums may be overwritten */
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int k = k0 + u * TR_T;
        if (k >= kend) continue;
        th[k] = *train_param(s, k);
        m[k] = mk[u];
        v[k] = vk[u];
    }
}

/* Cross-entropy of samples idx[0 .. count) with outputs pall[k], one FP64 partial sum per
 * block (summed in block order on the host). */
constexpr int LOSS_BLOCKS = 304, LOSS_T = 128;
__global__ void __launch_bounds__(LOSS_T) loss_kernel(const float *__restrict__ pall, const float *__restrict__ Y,
                                                      const int *__restrict__ idx, int count, double *__restrict__ part)
{
    __shared__ double sh[LOSS_T];
    double l = 0.0;
    for (int k = blockIdx.x * LOSS_T + threadIdx.x; k < count; k += LOSS_BLOCKS * LOSS_T) {
        const double y = (double)Y[idx[k]], pc = fmin(fmax((double)pall[k], 1e-30), 1.0 - 1e-7);
        if (y != 0.0) l -= y * log(pc);
        if (y != 1.0) l -= (1.0 - y) * log(1.0 - pc);
    }
    sh[threadIdx.x] = l;
    __syncthreads();
    for (int o = LOSS_T / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

/* BF16 copy of the weights used by inference. */
__global__ void to_bf16_kernel(const float *th, __nv_bfloat16 *wb)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < NPARAM) wb[k] = __float2bfloat16_rn(th[k]);
}

/* Inference on the tensor cores: mma.sync m16n8k16 with BF16 operands and FP32
 * accumulation. A warp takes 32 nodes at a time as two 16-node tiles (two independent
 * chains, one read of the weight fragments), or, of few nodes, one tile. Layer 1 is the 16 x 16 (8 features,
 * zero-padded) by 16 x 64 product; its GELU outputs are rounded to BF16 and, because
 * the accumulator fragment of two neighbouring 8-column output tiles has exactly the
 * element layout of one 16-wide operand fragment, feed layer 2 from registers; layer 2's
 * GELU outputs meet W3 in FP32 (a dot product over the 64 hidden units, finished across
 * the four lanes that share a row). The weight fragments are built in shared memory
 * once per block. A node with a non-finite feature gets p = NaN.
 *
 * What bounds it: the 128 GELUs of a node, on the FP32 and special-function units. They
 * are evaluated in pairs, as twice the GELU (the weights behind it are halved, which is exact):
 *   2 gelu(a) = (a + |a|) + y 2^P(y),   y = max(-|a|, -7),   2^P(-x) = erfc(x / sqrt 2),
 * with P a polynomial of degree 9 without a constant term (so that near zero, where P is
 * small, its rounding is too) in packed FP32 arithmetic, and one exp2 each: 8 instructions a
 * value against about 30 of the erf form. The coefficients are a weighted minimax fit
 * (iteratively reweighted least squares on Chebyshev nodes of [0, 7], each rounded to FP32 and
 * the rest fitted again) of log2 erfc, off by at most 3.7e-9 of GELU. a + |a| keeps the erf
 * form's values at NaN and the infinities (2 gelu(-inf) = NaN: the node has no p).
 * Against FP64, largest error, the erf form in FP32 in brackets: relative 1.8e-7 (1.3e-7) for
 * |a| < 0.25, 2.4e-7 (2.2e-7) to 1, 9.0e-8 (1.2e-7) for 1 < a < 9; absolute 4.4e-8 (6.5e-8) for
 * -2 < a < -1, 2.2e-8 (1.2e-7) below, 1.2e-11 (0) below -7. Rms: up to 1.6 times the erf form's
 * for -0.25 < a < 0, 1.1 times for 0 < a < 0.05 and -1 < a < -0.25, smaller elsewhere. (An earlier
 * fit to log2 of half the erfc, cut off at 5.75, was off by 9.8e-7 of the value near zero and by
 * 2.6e-8 below -5.75.)
 * 2 097 152 nodes: 345 us in the erf form, 201 with the earlier fit, 204 with this one. */
__device__ __forceinline__ float2 twice_gelu(float2 a)
{
    const float2 y = make_float2(fmaxf(-fabsf(a.x), -7.0f), fmaxf(-fabsf(a.y), -7.0f));
    constexpr float C[9] = {1.1511046886444092f,       -0.4592166244983673f,     0.05245400220155716f,
                            0.006968232337385416f,     2.4232918804045767e-05f,  -0.00026060346863232553f,
                            -6.681260128971189e-05f,   -8.086775778792799e-06f,  -4.048496009545488e-07f};
    float2 p = make_float2(C[8], C[8]);
#pragma unroll
    for (int k = 7; k >= 0; --k) p = __ffma2_rn(p, y, make_float2(C[k], C[k]));
    p = __fmul2_rn(p, y);
    float2 e;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.x) : "f"(p.x));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e.y) : "f"(p.y));
    return __ffma2_rn(y, e, make_float2(a.x + fabsf(a.x), a.y + fabsf(a.y)));
}

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2])
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&v);
}

__device__ __forceinline__ uint32_t pack_bf16_raw(__nv_bfloat16 lo, __nv_bfloat16 hi)
{
    __nv_bfloat162 v;
    v.x = lo;
    v.y = hi;
    return *reinterpret_cast<const uint32_t *>(&v);
}

/* (not inlined: rare, and 32 copies of it would not fit the instruction cache) */
__device__ __noinline__ uint32_t twice_gelu_erf_bf16(float2 a) { return pack_bf16(2.0f * gelu(a.x), 2.0f * gelu(a.y)); }

/* A pair of them rounded to BF16: a value that lies within 4 FP32 units of a rounding boundary
 * (one in 4096) is formed again in the erf form. For a > -1 the errors of the two forms add up
 * to less than that distance, so every value is rounded as the erf form rounds it; below, where
 * the erf form's own error is larger, the two may round apart. */
__device__ __forceinline__ uint32_t twice_gelu_bf16(float2 a)
{
    constexpr float D = 4.76837158e-7f;   /* 2^-21 */
    const float2 h = twice_gelu(a);
    const float2 lo = __fmul2_rn(h, make_float2(1.0f - D, 1.0f - D)), hi = __fmul2_rn(h, make_float2(1.0f + D, 1.0f + D));
    const uint32_t r = pack_bf16(lo.x, lo.y);
    return r == pack_bf16(hi.x, hi.y) ? r : twice_gelu_erf_bf16(a);
}

/* M tiles per warp pass: two, or one where that is all a resident warp gets */
template <int M>
__global__ void __launch_bounds__(128, 5) infer_mma_kernel(const __nv_bfloat16 *__restrict__ wb,
                                                           const float *__restrict__ norm,
                                                           const float *__restrict__ X, long long n,
                                                           float *__restrict__ p)
{
    /* operand fragments of the weights: B[k][n] of layer 1 is W1[n][k] (k < 8, zero
     * above), of layer 2 W2[n][k] / 2; fragment register r of lane l holds the rows
     * 2 (l % 4) + {0, 1} (+ 8 for r = 1) of column l / 4 */
    __shared__ uint32_t w1f[8][32];
    __shared__ uint2 w2f[4][8][32];
    __shared__ float2 b1s[NH / 2], b2s[NH / 2], w3s[NH / 2];
    __shared__ float nm[2 * NF], b3s;
    for (int k = threadIdx.x; k < 8 * 32; k += blockDim.x) {
        const int nt = k / 32, l = k % 32, col = 8 * nt + l / 4, row = 2 * (l % 4);
        w1f[nt][l] = pack_bf16_raw(wb[OFF_W1 + col * NF + row], wb[OFF_W1 + col * NF + row + 1]);
    }
    for (int k = threadIdx.x; k < 4 * 8 * 32; k += blockDim.x) {
        const int kt = k / 256, nt = (k / 32) % 8, l = k % 32;
        const int col = 8 * nt + l / 4, row = 16 * kt + 2 * (l % 4);
        const __nv_bfloat16 *w = wb + OFF_W2 + col * NH;
        auto half = [&](int r) { return 0.5f * __bfloat162float(w[r]); };   /* activations come doubled */
        w2f[kt][nt][l] = make_uint2(pack_bf16(half(row), half(row + 1)), pack_bf16(half(row + 8), half(row + 9)));
    }
    for (int k = threadIdx.x; k < NH / 2; k += blockDim.x) {
        auto two = [&](int off) { return make_float2(__bfloat162float(wb[off + 2 * k]), __bfloat162float(wb[off + 2 * k + 1])); };
        b1s[k] = two(OFF_B1);
        b2s[k] = two(OFF_B2);
        w3s[k] = __fmul2_rn(two(OFF_W3), make_float2(0.5f, 0.5f));
    }
    if (threadIdx.x < 2 * NF) nm[threadIdx.x] = norm[threadIdx.x];
    if (threadIdx.x == 0) b3s = __bfloat162float(wb[OFF_B3]);
    __syncthreads();

    const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
    const long long passes = (n + 16 * M - 1) / (16 * M);
    const long long stride = (long long)gridDim.x * (blockDim.x >> 5);
    /* features 2q, 2q + 1 of this lane's nodes (rows g, g + 8 of each tile) */
    float xr[2 * M][2];
    auto fetch = [&](long long t) {
#pragma unroll
        for (int k = 0; k < 2 * M; ++k) {
            const long long r = 16 * M * t + g + 8 * k;
#pragma unroll
            for (int e = 0; e < 2; ++e) xr[k][e] = r < n ? X[(long long)(2 * q + e) * n + r] : nm[2 * q + e];
        }
    };
    long long t = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (t < passes) fetch(t);
    for (; t < passes; t += stride) {
        /* layer-1 operands: normalised features (columns 8..15 zero) */
        uint32_t a1[M][2];
        bool ok[2 * M];
#pragma unroll
        for (int k = 0; k < 2 * M; ++k) {
            float x0 = (xr[k][0] - nm[2 * q]) / nm[NF + 2 * q], x1 = (xr[k][1] - nm[2 * q + 1]) / nm[NF + 2 * q + 1];
            /* a node is usable when all eight features are finite: the four lanes of a row
             * hold two each */
            const unsigned bad = __ballot_sync(0xffffffffu, !(isfinite(x0) && isfinite(x1)));
            ok[k] = !(bad & (0xfu << (4 * g)));
            if (!ok[k]) x0 = x1 = 0.0f;
            a1[k >> 1][k & 1] = pack_bf16(x0, x1);
        }
        if (t + stride < passes) fetch(t + stride);
        /* layer 1 -> GELU -> BF16 operand fragments of layer 2 */
        uint32_t a2[M][4][4];
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
            const uint32_t b[2] = {w1f[nt][lane], 0u};
            const float2 bias = b1s[4 * nt + q];
#pragma unroll
            for (int m = 0; m < M; ++m) {
                float c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                const uint32_t a[4] = {a1[m][0], a1[m][1], 0u, 0u};
                mma_bf16(c, a, b);
                const int kt = nt >> 1, hi = (nt & 1) * 2;
                a2[m][kt][hi] = twice_gelu_bf16(__fadd2_rn(make_float2(c[0], c[1]), bias));
                a2[m][kt][hi + 1] = twice_gelu_bf16(__fadd2_rn(make_float2(c[2], c[3]), bias));
            }
        }
        /* layer 2 -> GELU -> W3 dot product */
        float z[2 * M] = {};
#pragma unroll 2
        for (int nt = 0; nt < 8; ++nt) {
            float c[M][4] = {};
#pragma unroll
            for (int kt = 0; kt < 4; ++kt) {
                const uint2 w = w2f[kt][nt][lane];
                const uint32_t b[2] = {w.x, w.y};
#pragma unroll
                for (int m = 0; m < M; ++m) mma_bf16(c[m], a2[m][kt], b);
            }
            const float2 bias = b2s[4 * nt + q], w3 = w3s[4 * nt + q];
#pragma unroll
            for (int m = 0; m < M; ++m) {
                const float2 h0 = twice_gelu(__fadd2_rn(make_float2(c[m][0], c[m][1]), bias));
                const float2 h1 = twice_gelu(__fadd2_rn(make_float2(c[m][2], c[m][3]), bias));
                z[2 * m] = fmaf(h0.y, w3.y, fmaf(h0.x, w3.x, z[2 * m]));
                z[2 * m + 1] = fmaf(h1.y, w3.y, fmaf(h1.x, w3.x, z[2 * m + 1]));
            }
        }
#pragma unroll
        for (int k = 0; k < 2 * M; ++k) {
            z[k] += __shfl_xor_sync(0xffffffffu, z[k], 1);
            z[k] += __shfl_xor_sync(0xffffffffu, z[k], 2);
        }
        /* lane q of a row's four stores node k = q of its 2 M */
        float zq = z[0];
        bool okq = ok[0];
#pragma unroll
        for (int k = 1; k < 2 * M; ++k)
            if (q == k) {
                zq = z[k];
                okq = ok[k];
            }
        const long long r = 16 * M * t + g + 8 * q;
        if (q < 2 * M && r < n) p[r] = okq ? 1.0f / (1.0f + expf(-(zq + b3s))) : nanf("");
    }
}

}  // namespace lbm

/* ------------------------------------------------------------------ host -- */

struct lb_mlp {
    float *th = nullptr, *m = nullptr, *v = nullptr, *g = nullptr, *norm = nullptr;
    __nv_bfloat16 *wb = nullptr;
    int cap = 0;   /* batch capacity of the activation buffers */
    float *xn = nullptr, *a1 = nullptr, *h1 = nullptr, *a2 = nullptr, *h2 = nullptr, *p = nullptr, *dz = nullptr,
          *da1 = nullptr, *da2 = nullptr;
    double *loss = nullptr;
    /* training: order, outputs (one chunk of samples) and loss partials */
    int *idx = nullptr;
    float *pall = nullptr;
    double *lpart = nullptr;
    int idx_cap = 0, train_blocks = 0;
    int t = 0;
    lb_opts opts{};
    cudaStream_t stream = nullptr;
    std::vector<void *> owned;
};

namespace {

void *mlp_alloc(lb_mlp *M, size_t bytes)
{
    void *ptr = nullptr;
    if (M->opts.alloc && M->opts.free) ptr = M->opts.alloc(bytes, M->opts.alloc_user);
    else if (cudaMalloc(&ptr, bytes) != cudaSuccess) {
        cudaGetLastError();
        ptr = nullptr;
    }
    if (ptr) M->owned.push_back(ptr);
    return ptr;
}

void mlp_free_all(lb_mlp *M)
{
    if (M->stream) cudaStreamSynchronize(M->stream);
    for (void *ptr : M->owned) {
        if (M->opts.alloc && M->opts.free) M->opts.free(ptr, M->opts.alloc_user);
        else cudaFree(ptr);
    }
    M->owned.clear();
}

int mlp_err(int code, const std::string &msg)
{
    lbk::set_last_error(msg);
    return code;
}

int ensure_batch(lb_mlp *M, int B)
{
    if (B <= M->cap) return LB_OK;
    /* grow the activation buffers (old ones stay owned until destroy) */
    const size_t b = (size_t)B;
    M->xn = (float *)mlp_alloc(M, b * lbm::NF * 4);
    M->a1 = (float *)mlp_alloc(M, b * lbm::NH * 4);
    M->h1 = (float *)mlp_alloc(M, b * lbm::NH * 4);
    M->a2 = (float *)mlp_alloc(M, b * lbm::NH * 4);
    M->h2 = (float *)mlp_alloc(M, b * lbm::NH * 4);
    M->da1 = (float *)mlp_alloc(M, b * lbm::NH * 4);
    M->da2 = (float *)mlp_alloc(M, b * lbm::NH * 4);
    M->p = (float *)mlp_alloc(M, b * 4);
    M->dz = (float *)mlp_alloc(M, b * 4);
    if (!M->xn || !M->a1 || !M->h1 || !M->a2 || !M->h2 || !M->da1 || !M->da2 || !M->p || !M->dz)
        return mlp_err(LB_ERR_NOMEM, "lb_mlp: device allocation failed");
    M->cap = B;
    return LB_OK;
}

cudaLaunchConfig_t train_config(int nc, cudaLaunchAttribute *at, cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nc);
    cfg.blockDim = dim3(lbm::TR_T);
    cfg.dynamicSmemBytes = sizeof(lbm::TrainSmem);
    cfg.stream = st;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = nc;
    at->val.clusterDim.y = at->val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

/* blocks of the training cluster: 16 (beyond the portable size; a batch of 256 is then 16
 * samples a block) where the device takes such a cluster, else 8 */
int train_cluster()
{
    const int smem = (int)sizeof(lbm::TrainSmem);
    cudaLaunchAttribute at;
    int n = 0;
    if (cudaFuncSetAttribute(lbm::train_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess &&
        cudaFuncSetAttribute(lbm::train_kernel<16>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
        const cudaLaunchConfig_t cfg = train_config(16, &at, nullptr);
        if (cudaOccupancyMaxActiveClusters(&n, lbm::train_kernel<16>, &cfg) == cudaSuccess && n > 0) return 16;
    }
    cudaGetLastError();
    if (cudaFuncSetAttribute(lbm::train_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess) return 8;
    cudaGetLastError();
    return 0;
}

/* workspace of a training launch over `count` samples, and the kernel's shared memory */
int ensure_train(lb_mlp *M, int count)
{
    if (M->train_blocks == 0) M->train_blocks = train_cluster();
    if (M->train_blocks == 0) return mlp_err(LB_ERR_CUDA, "lb_mlp: the training kernel cannot be resident");
    if (!M->lpart) M->lpart = (double *)mlp_alloc(M, sizeof(double) * lbm::LOSS_BLOCKS);
    if (count > M->idx_cap) {
        /* grow (old buffers stay owned until destroy) */
        M->idx = (int *)mlp_alloc(M, (size_t)count * 4);
        M->pall = (float *)mlp_alloc(M, (size_t)count * 4);
        M->idx_cap = M->idx && M->pall ? count : 0;
    }
    if (!M->idx || !M->pall || !M->lpart) return mlp_err(LB_ERR_NOMEM, "lb_mlp: device allocation failed");
    return LB_OK;
}

/* forward + backward + weight gradients of the first B samples */
int batch_grad(lb_mlp *M, const float *x, const float *y, int64_t n, int B, bool want_loss)
{
    const int T = 128, nb = (B + T - 1) / T;
    if (want_loss && cudaMemsetAsync(M->loss, 0, sizeof(double), M->stream) != cudaSuccess)
        return mlp_err(LB_ERR_CUDA, "lb_mlp: memset failed");
    lbm::fwd_kernel<<<nb, T, 0, M->stream>>>(M->th, M->norm, x, (long long)n, B, M->xn, M->a1, M->h1, M->a2,
                                             M->h2, M->p);
    lbm::bwd_kernel<<<nb, T, 0, M->stream>>>(M->th, y, B, M->a1, M->a2, M->p, M->dz, M->da1, M->da2,
                                             want_loss ? M->loss : nullptr);
    lbm::wgrad_kernel<<<(lbm::NPARAM + 127) / 128, 128, 0, M->stream>>>(B, M->xn, M->h1, M->h2, M->dz, M->da1, M->da2,
                                                                        M->g);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? LB_OK : mlp_err(LB_ERR_CUDA, std::string("lb_mlp: ") + cudaGetErrorString(e));
}

}  // namespace

namespace lbk {

int mlp_infer_dev(lb_mlp *M, const float *x, int64_t n, float *p, void *stream)
{
    /* four warps per block, five blocks per SM resident (152 SMs): each warp walks its passes of
     * two 16-node tiles with a grid stride; of one tile where the warps outnumber the tiles, a
     * shorter chain (a call of 1 to 8000 nodes 17.4 -> 14.8 us, 40 000 nodes 20.1 -> 19.3; 16.1 to
     * 17.5 and 23 before two tiles shared a warp); the same values */
    constexpr long long RESIDENT = 152LL * 5;
    const long long tiles = (n + 15) / 16;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (tiles <= 4 * RESIDENT) {
        lbm::infer_mma_kernel<1><<<(unsigned)((tiles + 3) / 4), 128, 0, st>>>(M->wb, M->norm, x, (long long)n, p);
    } else {
        const unsigned blocks = (unsigned)std::min<long long>((tiles + 7) / 8, RESIDENT);
        lbm::infer_mma_kernel<2><<<blocks, 128, 0, st>>>(M->wb, M->norm, x, (long long)n, p);
    }
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? LB_OK : mlp_err(LB_ERR_CUDA, std::string("lb_mlp_infer: ") + cudaGetErrorString(e));
}

}  // namespace lbk

extern "C" {

int lb_mlp_create(const float *params, const float norm[16], const lb_opts *opts, lb_mlp **out)
{
    if (!params || !norm || !opts || !out) return mlp_err(LB_ERR_INVALID, "lb_mlp_create: null argument");
    for (int f = 0; f < lbm::NF; ++f)
        if (!(norm[lbm::NF + f] > 0.0f)) return mlp_err(LB_ERR_INVALID, "lb_mlp_create: feature scales must be positive");
    lb_mlp *M = new lb_mlp();
    M->opts = *opts;
    M->stream = static_cast<cudaStream_t>(opts->stream);
    M->th = (float *)mlp_alloc(M, lbm::NPARAM * 4);
    M->m = (float *)mlp_alloc(M, lbm::NPARAM * 4);
    M->v = (float *)mlp_alloc(M, lbm::NPARAM * 4);
    M->g = (float *)mlp_alloc(M, lbm::NPARAM * 4);
    M->wb = (__nv_bfloat16 *)mlp_alloc(M, lbm::NPARAM * 2);
    M->norm = (float *)mlp_alloc(M, 2 * lbm::NF * 4);
    M->loss = (double *)mlp_alloc(M, 256);
    if (!M->th || !M->m || !M->v || !M->g || !M->wb || !M->norm || !M->loss) {
        mlp_free_all(M);
        delete M;
        return mlp_err(LB_ERR_NOMEM, "lb_mlp_create: device allocation failed");
    }
    cudaError_t e = cudaMemcpyAsync(M->th, params, lbm::NPARAM * 4, cudaMemcpyHostToDevice, M->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(M->norm, norm, 2 * lbm::NF * 4, cudaMemcpyHostToDevice, M->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(M->m, 0, lbm::NPARAM * 4, M->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(M->v, 0, lbm::NPARAM * 4, M->stream);
    if (e == cudaSuccess) {
        lbm::to_bf16_kernel<<<(lbm::NPARAM + 255) / 256, 256, 0, M->stream>>>(M->th, M->wb);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(M->stream);
    if (e != cudaSuccess) {
        mlp_free_all(M);
        delete M;
        return mlp_err(LB_ERR_CUDA, std::string("lb_mlp_create: ") + cudaGetErrorString(e));
    }
    *out = M;
    return LB_OK;
}

int lb_mlp_grad(lb_mlp *M, const float *x, const float *y, int64_t n, float *grad, double *loss)
{
    if (!M || !x || !y || !grad || n < 1 || n > (1 << 20)) return mlp_err(LB_ERR_INVALID, "lb_mlp_grad: bad argument");
    if (int e = ensure_batch(M, (int)n)) return e;
    if (int e = batch_grad(M, x, y, n, (int)n, true)) return e;
    cudaError_t ce = cudaMemcpyAsync(grad, M->g, lbm::NPARAM * 4, cudaMemcpyDeviceToHost, M->stream);
    double l = 0.0;
    if (ce == cudaSuccess) ce = cudaMemcpyAsync(&l, M->loss, sizeof(double), cudaMemcpyDeviceToHost, M->stream);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(M->stream);
    if (ce != cudaSuccess) return mlp_err(LB_ERR_CUDA, std::string("lb_mlp_grad: ") + cudaGetErrorString(ce));
    if (loss) *loss = l;
    return LB_OK;
}

int lb_mlp_train(lb_mlp *M, const float *x, const float *y, int64_t n, int32_t epochs, int32_t batch, float lr,
                 uint64_t seed, double *last_epoch_loss)
{
    if (!M || !x || !y || n < 1 || epochs < 1 || batch < 1 || batch > 65536 || !(lr > 0.0f))
        return mlp_err(LB_ERR_INVALID, "lb_mlp_train: bad argument");
    /* whole batches of at most TRAIN_CHUNK samples (one batch at least) per launch: the order
     * and the outputs of a launch's samples are the workspace */
    constexpr int64_t TRAIN_CHUNK = 1 << 18;
    const int64_t chunk = std::min<int64_t>(n, std::max<int64_t>(1, TRAIN_CHUNK / batch) * batch);
    if (int e = ensure_train(M, (int)chunk)) return e;
    std::vector<int> perm((size_t)n);
    for (int64_t k = 0; k < n; ++k) perm[(size_t)k] = (int)k;
    std::mt19937_64 rng(seed);
    double eloss = 0.0;
    for (int ep = 0; ep < epochs; ++ep) {
        for (int64_t k = n - 1; k > 0; --k) std::swap(perm[(size_t)k], perm[(size_t)(rng() % (uint64_t)(k + 1))]);
        const bool last_epoch = ep == epochs - 1;
        for (int64_t s0 = 0; s0 < n; s0 += chunk) {
            const int cnt = (int)std::min<int64_t>(chunk, n - s0);
            if (cudaMemcpyAsync(M->idx, perm.data() + s0, (size_t)cnt * 4, cudaMemcpyHostToDevice, M->stream) != cudaSuccess)
                return mlp_err(LB_ERR_CUDA, "lb_mlp_train: copy failed");
            cudaLaunchAttribute at;
            const cudaLaunchConfig_t cfg = train_config(M->train_blocks, &at, M->stream);
            float *pall = last_epoch ? M->pall : nullptr;
            const cudaError_t le = cudaLaunchKernelEx(
                &cfg, M->train_blocks == 16 ? lbm::train_kernel<16> : lbm::train_kernel<8>, M->th, M->m, M->v,
                (const float *)M->norm, x, (long long)n, y, (const int *)M->idx, cnt, (int)batch, M->t, lr, pall);
            if (le != cudaSuccess) return mlp_err(LB_ERR_CUDA, std::string("lb_mlp_train: ") + cudaGetErrorString(le));
            M->t += (cnt + batch - 1) / batch;
            if (last_epoch) {
                double part[lbm::LOSS_BLOCKS];
                lbm::loss_kernel<<<lbm::LOSS_BLOCKS, lbm::LOSS_T, 0, M->stream>>>(M->pall, y, M->idx, cnt, M->lpart);
                if (cudaMemcpyAsync(part, M->lpart, sizeof(part), cudaMemcpyDeviceToHost, M->stream) != cudaSuccess ||
                    cudaStreamSynchronize(M->stream) != cudaSuccess)
                    return mlp_err(LB_ERR_CUDA, "lb_mlp_train: copy failed");
                for (double l : part) eloss += l;
            }
        }
        /* keep perm as it is until its last upload has finished */
        if (cudaStreamSynchronize(M->stream) != cudaSuccess) return mlp_err(LB_ERR_CUDA, "lb_mlp_train: sync failed");
    }
    lbm::to_bf16_kernel<<<(lbm::NPARAM + 255) / 256, 256, 0, M->stream>>>(M->th, M->wb);
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(M->stream) != cudaSuccess)
        return mlp_err(LB_ERR_CUDA, "lb_mlp_train: kernel failed");
    if (last_epoch_loss) *last_epoch_loss = eloss / (double)n;
    return LB_OK;
}

int lb_mlp_adam_step(lb_mlp *M, const float *x, const float *y, int64_t n, float lr)
{
    if (!M || !x || !y || n < 1 || n > (1 << 20)) return mlp_err(LB_ERR_INVALID, "lb_mlp_adam_step: bad argument");
    if (int e = ensure_batch(M, (int)n)) return e;
    if (int e = batch_grad(M, x, y, n, (int)n, false)) return e;
    M->t += 1;
    lbm::adam_kernel<<<(lbm::NPARAM + 127) / 128, 128, 0, M->stream>>>(M->th, M->m, M->v, M->g, M->t, lr, 0.9f, 0.999f,
                                                                      1e-8f);
    lbm::to_bf16_kernel<<<(lbm::NPARAM + 255) / 256, 256, 0, M->stream>>>(M->th, M->wb);
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(M->stream) != cudaSuccess)
        return mlp_err(LB_ERR_CUDA, "lb_mlp_adam_step: kernel failed");
    return LB_OK;
}

int lb_mlp_get_params(lb_mlp *M, float *params)
{
    if (!M || !params) return mlp_err(LB_ERR_INVALID, "lb_mlp_get_params: null argument");
    if (cudaMemcpyAsync(params, M->th, lbm::NPARAM * 4, cudaMemcpyDeviceToHost, M->stream) != cudaSuccess ||
        cudaStreamSynchronize(M->stream) != cudaSuccess)
        return mlp_err(LB_ERR_CUDA, "lb_mlp_get_params: copy failed");
    return LB_OK;
}

int lb_mlp_infer(lb_mlp *M, const float *x, int64_t n, float *p)
{
    if (!M || !x || !p || n < 1) return mlp_err(LB_ERR_INVALID, "lb_mlp_infer: bad argument");
    if (int e = lbk::mlp_infer_dev(M, x, n, p, M->stream)) return e;
    return cudaStreamSynchronize(M->stream) == cudaSuccess ? LB_OK : mlp_err(LB_ERR_CUDA, "lb_mlp_infer: sync failed");
}

void lb_mlp_destroy(lb_mlp *M)
{
    if (!M) return;
    mlp_free_all(M);
    delete M;
}

}  // extern "C"
