// mlp.cu -- the plan-cost model: a 3-layer perceptron F -> H -> H -> 1 with
// exact GELU, trained on measured plan timings (log run time, MSE loss, Adam)
// entirely by the kernels below.  No counterpart in the paper, which leaves
// the choice of decomposition to the user; the model ranks candidate plans
// for shapes it has not timed, and exhaustive autotuning stays the fallback.
//
// Parameters are one flat float array: W1 (H x F), b1 (H), W2 (H x H), b2 (H),
// W3 (1 x H), b3 (1), row-major.  Activations are row-major (samples x units).
#include <cooperative_groups.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <random>
#include <vector>

#include "capi_internal.h"

namespace fft3 {

struct MlpLayout {
    int F, H;
    int w1, b1, w2, b2, w3, b3, total;
    explicit MlpLayout(int f = 0, int h = 0) : F(f), H(h)
    {
        w1 = 0;
        b1 = w1 + H * F;
        w2 = b1 + H;
        b2 = w2 + H * H;
        w3 = b2 + H;
        b3 = w3 + H;
        total = b3 + 1;
    }
};

__device__ __forceinline__ float gelu_f(float x) { return 0.5f * x * (1.f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float x)
{
    const float Phi = 0.5f * (1.f + erff(x * 0.70710678118654752f));
    const float phi = 0.39894228040143268f * expf(-0.5f * x * x);
    return Phi + x * phi;
}

// ------------------------------------------------------ fused gradient -- //
// Loss and gradient of a minibatch in one launch, for the widths the model is
// used at (H = 32, 64 or 128, F <= 64): the layer-by-layer kernels below took
// nine launches of 2 to 10 us each (16 steps of 128 samples, F = 32, H = 64:
// 1335 us; with this kernel 220 us, a third of it launches and the copies of the
// parameters).  What bounds it: latency, a minibatch being a few microseconds of
// work for a handful of SMs.
// A cluster of 8 blocks holds a copy of the parameters each and takes chunks of
// 16 samples in turn, two samples per warp.  A lane owns the units n = lane + 32 j:
// the pre-activations stay in its registers from the forward to the backward
// pass, and only h1, dz1, dz2 and the inputs go through shared memory, for the
// weight gradients, whose sums over all chunks stay in registers.  At the end
// every block sums its share of the parameters over the cluster's shared
// memories.  More than 128 samples are spread over several clusters whose sums a
// second kernel adds.  All sums run in a fixed order.
constexpr int kGradCluster = 8, kGradChunk = 16, kGradThreads = 256, kGradMaxF = 64, kGradMaxClusters = 16;

__host__ __device__ constexpr int grad_pitch(int f) { return (f + 3) / 4 * 4 + 4; } // rows read as float4

// Dynamic shared memory, in floats.
__host__ __device__ constexpr int grad_smem_floats(int F, int H, int params)
{
    return H * (F | 1) + H * (H + 1) + 3 * H + 4           // W1, W2 (odd pitches), b1, b2, W3, b3
           + kGradChunk * (grad_pitch(F) + 3 * (H + 4))     // inputs; h1, dz2, dz1
           + 8 * (3 * H + 2)                                // per-warp sums of db1, db2, dW3, db3, loss
           + params + 4;                                    // the block's gradient, then its loss
}

template <int H>
__global__ void __cluster_dims__(kGradCluster, 1, 1) __launch_bounds__(kGradThreads)
    k_mlp_grad_fused(const float *p, MlpLayout L, const float *X, const float *y, const int *idx, int B, float *g0,
                     float *g1, float *loss0, float *loss1)
{
    namespace cg = cooperative_groups;
    constexpr int J = H / 32, NW = H / 8; // units per lane; rows of a weight gradient per warp
    extern __shared__ __align__(16) float sm[];
    const int F = L.F, FP = F | 1, XP = grad_pitch(F), KF = F > 32 ? 2 : 1;
    constexpr int HP = H + 4;
    float *xs = sm, *h1 = xs + kGradChunk * XP, *dz2 = h1 + kGradChunk * HP, *dz1 = dz2 + kGradChunk * HP;
    float *w1 = dz1 + kGradChunk * HP, *w2 = w1 + H * FP, *b1 = w2 + H * (H + 1), *b2 = b1 + H, *w3 = b2 + H,
          *b3 = w3 + H, *red = b3 + 4, *grad = red + 8 * (3 * H + 2);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    asm volatile("griddepcontrol.wait;" ::: "memory"); // the Adam step before may still run
    // a warp copies rows n = warp, warp + 8, ... (every load of a row set in flight at once)
#pragma unroll
    for (int i = 0; i < NW; ++i) {
        const int n = warp + 8 * i;
#pragma unroll
        for (int j = 0; j < J; ++j)
            w2[n * (H + 1) + lane + 32 * j] = p[L.w2 + n * H + lane + 32 * j];
#pragma unroll
        for (int j = 0; j < 2; ++j)
            if (lane + 32 * j < F)
                w1[n * FP + lane + 32 * j] = p[L.w1 + n * F + lane + 32 * j];
    }
    for (int i = tid; i < H; i += kGradThreads) {
        b1[i] = p[L.b1 + i];
        b2[i] = p[L.b2 + i];
        w3[i] = p[L.w3 + i];
    }
    if (tid == 0)
        b3[0] = p[L.b3];
    float a1[NW][2] = {}, a2[NW][J] = {}; // sums of dW1 and dW2: row warp * NW + i, column lane + 32 j
    float ab1[J] = {}, ab2[J] = {}, aw3[J] = {}, ab3 = 0.f, al = 0.f;
    const int chunks = (B + kGradChunk - 1) / kGradChunk;
    for (int c = blockIdx.x; c < chunks; c += gridDim.x) {
        __syncthreads(); // parameters loaded, or the previous chunk's sums done
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int r = 2 * warp + q, b = c * kGradChunk + r;
            const int64_t row = b < B ? (int64_t)(idx ? idx[b] : b) * F : 0;
            for (int k = lane; k < XP; k += 32)
                xs[r * XP + k] = b < B && k < F ? X[row + k] : 0.f;
        }
        __syncthreads();
        // forward: samples s0 and s0 + 1, units lane + 32 j
        const int s0 = 2 * warp;
        float z1[2][J], z2[2][J];
#pragma unroll
        for (int j = 0; j < J; ++j)
            z1[0][j] = z1[1][j] = b1[lane + 32 * j];
#pragma unroll 8
        for (int k = 0; k < F; ++k) {
            const float x0 = xs[s0 * XP + k], x1 = xs[(s0 + 1) * XP + k];
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const float w = w1[(lane + 32 * j) * FP + k];
                z1[0][j] = fmaf(x0, w, z1[0][j]);
                z1[1][j] = fmaf(x1, w, z1[1][j]);
            }
        }
#pragma unroll
        for (int j = 0; j < J; ++j) {
            h1[s0 * HP + lane + 32 * j] = gelu_f(z1[0][j]);
            h1[(s0 + 1) * HP + lane + 32 * j] = gelu_f(z1[1][j]);
            z2[0][j] = z2[1][j] = b2[lane + 32 * j];
        }
        __syncwarp();
#pragma unroll 4
        for (int k = 0; k < H; k += 4) {
            const float4 q0 = *reinterpret_cast<const float4 *>(h1 + s0 * HP + k);
            const float4 q1 = *reinterpret_cast<const float4 *>(h1 + (s0 + 1) * HP + k);
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const float *w = w2 + (lane + 32 * j) * (H + 1) + k;
                z2[0][j] = fmaf(q0.w, w[3], fmaf(q0.z, w[2], fmaf(q0.y, w[1], fmaf(q0.x, w[0], z2[0][j]))));
                z2[1][j] = fmaf(q1.w, w[3], fmaf(q1.z, w[2], fmaf(q1.y, w[1], fmaf(q1.x, w[0], z2[1][j]))));
            }
        }
        // output, loss, dz2 = g3 W3 gelu'(z2)
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            float h2[J], o = 0.f;
#pragma unroll
            for (int j = 0; j < J; ++j) {
                h2[j] = gelu_f(z2[s][j]);
                o = fmaf(h2[j], w3[lane + 32 * j], o);
            }
#pragma unroll
            for (int m = 16; m > 0; m >>= 1)
                o += __shfl_xor_sync(0xffffffffu, o, m);
            const int b = c * kGradChunk + s0 + s;
            const float d = b < B ? o + b3[0] - y[idx ? idx[b] : b] : 0.f;
            const float g = 2.f * d / (float)B;
            al += d * d / (float)B;
            ab3 += g;
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const int n = lane + 32 * j;
                aw3[j] = fmaf(g, h2[j], aw3[j]);
                const float dz = g * w3[n] * gelu_grad_f(z2[s][j]);
                ab2[j] += dz;
                dz2[(s0 + s) * HP + n] = dz;
            }
        }
        __syncwarp();
        // dz1 = (dz2 W2) gelu'(z1)
        float d1[2][J] = {};
#pragma unroll 4
        for (int n = 0; n < H; n += 4) {
            const float4 q0 = *reinterpret_cast<const float4 *>(dz2 + s0 * HP + n);
            const float4 q1 = *reinterpret_cast<const float4 *>(dz2 + (s0 + 1) * HP + n);
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const float *w = w2 + n * (H + 1) + lane + 32 * j;
                const float wa = w[0], wb = w[H + 1], wc = w[2 * (H + 1)], wd = w[3 * (H + 1)];
                d1[0][j] = fmaf(q0.w, wd, fmaf(q0.z, wc, fmaf(q0.y, wb, fmaf(q0.x, wa, d1[0][j]))));
                d1[1][j] = fmaf(q1.w, wd, fmaf(q1.z, wc, fmaf(q1.y, wb, fmaf(q1.x, wa, d1[1][j]))));
            }
        }
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const float dz = d1[s][j] * gelu_grad_f(z1[s][j]);
                ab1[j] += dz;
                dz1[(s0 + s) * HP + lane + 32 * j] = dz;
            }
        __syncthreads();
        // weight gradients over the chunk's samples
#pragma unroll 4
        for (int s = 0; s < kGradChunk; ++s) {
            float hv[J], xv[2];
#pragma unroll
            for (int j = 0; j < J; ++j)
                hv[j] = h1[s * HP + lane + 32 * j];
            xv[0] = lane < F ? xs[s * XP + lane] : 0.f;
            xv[1] = KF > 1 && lane + 32 < F ? xs[s * XP + lane + 32] : 0.f;
#pragma unroll
            for (int i = 0; i < NW; i += 4) {
                const float4 e = *reinterpret_cast<const float4 *>(dz2 + s * HP + warp * NW + i);
                const float4 f = *reinterpret_cast<const float4 *>(dz1 + s * HP + warp * NW + i);
                const float ev[4] = {e.x, e.y, e.z, e.w}, fv[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
#pragma unroll
                    for (int j = 0; j < J; ++j)
                        a2[i + u][j] = fmaf(ev[u], hv[j], a2[i + u][j]);
                    a1[i + u][0] = fmaf(fv[u], xv[0], a1[i + u][0]);
                    a1[i + u][1] = fmaf(fv[u], xv[1], a1[i + u][1]);
                }
            }
        }
    }
    // the block's sums, in the parameters' order
#pragma unroll
    for (int i = 0; i < NW; ++i) {
        const int n = warp * NW + i;
#pragma unroll
        for (int j = 0; j < J; ++j)
            grad[L.w2 + n * H + lane + 32 * j] = a2[i][j];
#pragma unroll
        for (int j = 0; j < 2; ++j)
            if (lane + 32 * j < F)
                grad[L.w1 + n * F + lane + 32 * j] = a1[i][j];
    }
    float *rw = red + warp * (3 * H + 2);
#pragma unroll
    for (int j = 0; j < J; ++j) {
        rw[lane + 32 * j] = ab1[j];
        rw[H + lane + 32 * j] = ab2[j];
        rw[2 * H + lane + 32 * j] = aw3[j];
    }
    if (lane == 0) {
        rw[3 * H] = ab3;
        rw[3 * H + 1] = al;
    }
    __syncthreads();
    for (int i = tid; i < 3 * H + 2; i += kGradThreads) {
        float v = 0.f;
        for (int w = 0; w < 8; ++w)
            v += red[w * (3 * H + 2) + i];
        const int at = i < H ? L.b1 + i : i < 2 * H ? L.b2 + i - H : i < 3 * H ? L.w3 + i - 2 * H
                     : i == 3 * H ? L.b3 : L.total;
        grad[at] = v;
    }
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    // this block's share of the parameters (and the loss at the end) over the cluster; with several
    // clusters g0 is their workspace, L.total + 1 values each
    const int rank = (int)cl.block_rank(), cluster = blockIdx.x / kGradCluster;
    const bool alone = gridDim.x == kGradCluster;
    for (int i = rank * kGradThreads + tid; i <= L.total; i += kGradCluster * kGradThreads) {
        float v = 0.f;
        for (int r = 0; r < kGradCluster; ++r)
            v += *cl.map_shared_rank(grad + i, r);
        if (!alone) {
            g0[(int64_t)cluster * (L.total + 1) + i] = v;
        } else if (i < L.total) {
            g0[i] = v;
            if (g1)
                g1[i] = v;
        } else {
            *loss0 = v;
            if (loss1)
                *loss1 = v;
        }
    }
    cl.sync(); // the other blocks have read this one's sums
}

// Sums of the clusters' gradients.
__global__ void k_mlp_grad_sum(const float *ws, int clusters, int total, float *g0, float *g1, float *loss0, float *loss1)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i > total)
        return;
    float v = 0.f;
    for (int c = 0; c < clusters; ++c)
        v += ws[(int64_t)c * (total + 1) + i];
    if (i < total) {
        g0[i] = v;
        if (g1)
            g1[i] = v;
    } else {
        *loss0 = v;
        if (loss1)
            *loss1 = v;
    }
}

// Z[b, n] = sum_k A[b, k] W[n, k] + bias[n];  H = act ? gelu(Z) : Z.
__global__ void k_mlp_linear(const float *A, const float *W, const float *bias, float *Z, float *Hout, int B, int K,
                             int N, int act)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= B * N)
        return;
    const int b = i / N, n = i - b * N;
    float s = bias[n];
    for (int k = 0; k < K; ++k)
        s = fmaf(A[b * K + k], W[n * K + k], s);
    Z[i] = s;
    if (Hout)
        Hout[i] = act ? gelu_f(s) : s;
}

// g[b] = (2/B) (pred[b] - y[b]); loss += sum (pred - y)^2 / B.
__global__ void k_mlp_mse(const float *pred, const float *y, int B, float *g, float *loss)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    float d = 0.f;
    if (i < B) {
        d = pred[i] - y[i];
        g[i] = 2.f * d / (float)B;
    }
    float v = d * d / (float)B;
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0 && loss)
        atomicAdd(loss, v);
}

// dW[n, k] = sum_b dZ[b, n] A[b, k]; db[n] = sum_b dZ[b, n] (k == 0 threads).
__global__ void k_mlp_wgrad(const float *dZ, const float *A, int B, int K, int N, float *dW, float *db)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N * (K + 1))
        return;
    const int n = i / (K + 1), k = i - n * (K + 1);
    float s = 0.f;
    if (k < K) {
        for (int b = 0; b < B; ++b)
            s = fmaf(dZ[b * N + n], A[b * K + k], s);
        dW[n * K + k] = s;
    } else {
        for (int b = 0; b < B; ++b)
            s += dZ[b * N + n];
        db[n] = s;
    }
}

// dZprev[b, k] = (sum_n dZ[b, n] W[n, k]) * gelu'(Zprev[b, k]).
__global__ void k_mlp_backprop(const float *dZ, const float *W, const float *Zprev, int B, int K, int N, float *dZprev)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= B * K)
        return;
    const int b = i / K, k = i - b * K;
    float s = 0.f;
    for (int n = 0; n < N; ++n)
        s = fmaf(dZ[b * N + n], W[n * K + k], s);
    dZprev[i] = s * gelu_grad_f(Zprev[i]);
}

// Adam (Kingma & Ba) with bias correction; t is the 1-based step.
__global__ void k_mlp_adam(float *p, const float *g, float *m, float *v, int n, float lr, float b1, float b2,
                           float eps, float c1, float c2)
{
    asm volatile("griddepcontrol.wait;" ::: "memory"); // launched while the gradient's kernel drains
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

__global__ void k_mlp_gather(const float *X, const float *y, const int *idx, int B, int F, float *Xb, float *yb)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= B * (F + 1))
        return;
    const int b = i / (F + 1), f = i - b * (F + 1);
    const int s = idx[b];
    if (f < F)
        Xb[b * F + f] = X[s * F + f];
    else
        yb[b] = y[s];
}

} // namespace fft3

using namespace fft3;

struct fft3_mlp_s {
    MlpLayout L;
    float *d_p = nullptr, *d_g = nullptr, *d_m = nullptr, *d_v = nullptr;
    // activations for up to cap samples
    int cap = 0;
    float *z1 = nullptr, *h1 = nullptr, *z2 = nullptr, *h2 = nullptr, *z3 = nullptr, *g3 = nullptr, *g2 = nullptr,
          *g1 = nullptr, *loss = nullptr;
    int step = 0;
    float *grad_ws = nullptr; // gradients of several clusters (k_mlp_grad_fused)
};

static void mlp_free_acts(fft3_mlp_s *m)
{
    float *ptrs[] = {m->z1, m->h1, m->z2, m->h2, m->z3, m->g3, m->g2, m->g1};
    for (float *p : ptrs)
        cudaFree(p);
    m->z1 = m->h1 = m->z2 = m->h2 = m->z3 = m->g3 = m->g2 = m->g1 = nullptr;
    m->cap = 0;
}

static int mlp_reserve(fft3_mlp_s *m, int B)
{
    if (B <= m->cap)
        return FFT3_OK;
    mlp_free_acts(m);
    const int H = m->L.H;
    size_t bh = (size_t)B * H * sizeof(float), b1 = (size_t)B * sizeof(float);
    if (cudaMalloc(&m->z1, bh) || cudaMalloc(&m->h1, bh) || cudaMalloc(&m->z2, bh) || cudaMalloc(&m->h2, bh) ||
        cudaMalloc(&m->z3, b1) || cudaMalloc(&m->g3, b1) || cudaMalloc(&m->g2, bh) || cudaMalloc(&m->g1, bh)) {
        cudaGetLastError();
        mlp_free_acts(m);
        return fail(FFT3_ERR_OOM, "MLP activation allocation failed");
    }
    m->cap = B;
    return FFT3_OK;
}

static inline int nblk(int n) { return std::max(1, (n + 255) / 256); }

static int mlp_fwd(fft3_mlp_s *m, const float *X, int B, cudaStream_t st)
{
    const MlpLayout &L = m->L;
    const float *p = m->d_p;
    k_mlp_linear<<<nblk(B * L.H), 256, 0, st>>>(X, p + L.w1, p + L.b1, m->z1, m->h1, B, L.F, L.H, 1);
    k_mlp_linear<<<nblk(B * L.H), 256, 0, st>>>(m->h1, p + L.w2, p + L.b2, m->z2, m->h2, B, L.H, L.H, 1);
    k_mlp_linear<<<nblk(B), 256, 0, st>>>(m->h2, p + L.w3, p + L.b3, m->z3, nullptr, B, L.H, 1, 0);
    CUDA_TRY(cudaGetLastError());
    return FFT3_OK;
}

// Loss and gradient of the MSE over B samples into m->d_g (and m->loss).
static int mlp_bwd(fft3_mlp_s *m, const float *X, const float *y, int B, cudaStream_t st)
{
    const MlpLayout &L = m->L;
    const float *p = m->d_p;
    float *g = m->d_g;
    CUDA_TRY(cudaMemsetAsync(m->loss, 0, sizeof(float), st));
    k_mlp_mse<<<nblk(B), 256, 0, st>>>(m->z3, y, B, m->g3, m->loss);
    k_mlp_wgrad<<<nblk(1 * (L.H + 1)), 256, 0, st>>>(m->g3, m->h2, B, L.H, 1, g + L.w3, g + L.b3);
    k_mlp_backprop<<<nblk(B * L.H), 256, 0, st>>>(m->g3, p + L.w3, m->z2, B, L.H, 1, m->g2);
    k_mlp_wgrad<<<nblk(L.H * (L.H + 1)), 256, 0, st>>>(m->g2, m->h1, B, L.H, L.H, g + L.w2, g + L.b2);
    k_mlp_backprop<<<nblk(B * L.H), 256, 0, st>>>(m->g2, p + L.w2, m->z1, B, L.H, L.H, m->g1);
    k_mlp_wgrad<<<nblk(L.H * (L.F + 1)), 256, 0, st>>>(m->g1, X, B, L.F, L.H, g + L.w1, g + L.b1);
    CUDA_TRY(cudaGetLastError());
    return FFT3_OK;
}

static const void *grad_fused_kernel(const MlpLayout &L)
{
    if (L.F > kGradMaxF || grad_smem_floats(L.F, L.H, L.total) * sizeof(float) > (size_t)kSmemLimit)
        return nullptr;
    return L.H == 32    ? (const void *)&k_mlp_grad_fused<32>
           : L.H == 64  ? (const void *)&k_mlp_grad_fused<64>
           : L.H == 128 ? (const void *)&k_mlp_grad_fused<128>
                        : nullptr;
}

// A launch that may start while the kernel before it on the stream drains (its
// kernel waits: griddepcontrol.wait).
static cudaError_t launch_after(const void *f, int grid, int block, int smem, cudaStream_t st, void **args)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, f, args);
}

// Loss and gradient of B samples (rows idx[b] of X and y, or rows b) into m->d_g
// and m->loss, and into g1 and loss1 unless null.
static int mlp_gradient(fft3_mlp_s *m, const float *X, const float *y, const int *idx, int B, float *g1, float *loss1,
                        cudaStream_t st)
{
    const MlpLayout &L = m->L;
    const void *f = grad_fused_kernel(L);
    // a chunk per block while the clusters last (a chunk takes 5 us, the second kernel 3)
    const int chunks = (B + kGradChunk - 1) / kGradChunk;
    int clusters = std::min(kGradMaxClusters, (chunks + kGradCluster - 1) / kGradCluster);
    float *g0 = clusters > 1 ? m->grad_ws : m->d_g;
    const float *p = m->d_p;
    float *loss0 = m->loss;
    int total = L.total;
    MlpLayout lay = L;
    void *args[] = {&p, &lay, &X, &y, &idx, &B, &g0, &g1, &loss0, &loss1};
    CUDA_TRY(launch_after(f, clusters * kGradCluster, kGradThreads,
                          grad_smem_floats(L.F, L.H, L.total) * (int)sizeof(float), st, args));
    if (clusters > 1) {
        float *out = m->d_g;
        void *sargs[] = {&g0, &clusters, &total, &out, &g1, &loss0, &loss1};
        CUDA_TRY(launch_after((const void *)&k_mlp_grad_sum, nblk(total + 1), 256, 0, st, sargs));
    }
    return FFT3_OK;
}

extern "C" {

int fft3_mlp_create(fft3_mlp *out, int n_features, int hidden, unsigned long long seed)
{
    if (!out || n_features < 1 || hidden < 1 || n_features > 4096 || hidden > 4096)
        return fail(FFT3_ERR_INVALID_ARG, "bad MLP shape");
    *out = nullptr;
    int dev = 0;
    int rc = check_device(&dev);
    if (rc)
        return rc;
    auto *m = new (std::nothrow) fft3_mlp_s();
    if (!m)
        return fail(FFT3_ERR_OOM, "host allocation failed");
    m->L = MlpLayout(n_features, hidden);
    const size_t bytes = (size_t)m->L.total * sizeof(float);
    if (cudaMalloc(&m->d_p, bytes) || cudaMalloc(&m->d_g, bytes) || cudaMalloc(&m->d_m, bytes) ||
        cudaMalloc(&m->d_v, bytes) || cudaMalloc(&m->loss, sizeof(float))) {
        cudaGetLastError();
        fft3_mlp_destroy(m);
        return fail(FFT3_ERR_OOM, "MLP allocation failed");
    }
    if (const void *f = grad_fused_kernel(m->L)) {
        const int smem = grad_smem_floats(n_features, hidden, m->L.total) * (int)sizeof(float);
        if (cudaMalloc(&m->grad_ws, (size_t)kGradMaxClusters * (m->L.total + 1) * sizeof(float)) ||
            cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) {
            cudaGetLastError();
            fft3_mlp_destroy(m);
            return fail(FFT3_ERR_OOM, "MLP allocation failed");
        }
    }
    // He-style initialisation from a seeded generator on the host
    std::mt19937_64 rng(seed);
    std::vector<float> p(m->L.total, 0.f);
    auto fill = [&](int off, int rows, int cols) {
        std::normal_distribution<double> nd(0.0, std::sqrt(2.0 / cols));
        for (int i = 0; i < rows * cols; ++i)
            p[off + i] = (float)nd(rng);
    };
    fill(m->L.w1, hidden, n_features);
    fill(m->L.w2, hidden, hidden);
    fill(m->L.w3, 1, hidden);
    cudaMemcpy(m->d_p, p.data(), bytes, cudaMemcpyHostToDevice);
    cudaMemset(m->d_m, 0, bytes);
    cudaMemset(m->d_v, 0, bytes);
    cudaMemset(m->d_g, 0, bytes);
    *out = m;
    return FFT3_OK;
}

int fft3_mlp_destroy(fft3_mlp m)
{
    if (!m)
        return fail(FFT3_ERR_INVALID_ARG, "null model");
    mlp_free_acts(m);
    cudaFree(m->d_p);
    cudaFree(m->d_g);
    cudaFree(m->d_m);
    cudaFree(m->d_v);
    cudaFree(m->loss);
    cudaFree(m->grad_ws);
    delete m;
    return FFT3_OK;
}

int fft3_mlp_num_params(fft3_mlp m) { return m ? m->L.total : fail(FFT3_ERR_INVALID_ARG, "null model"); }

int fft3_mlp_set_params(fft3_mlp m, const float *h_params)
{
    if (!m || !h_params)
        return fail(FFT3_ERR_INVALID_ARG, "null argument");
    CUDA_TRY(cudaMemcpy(m->d_p, h_params, (size_t)m->L.total * 4, cudaMemcpyHostToDevice));
    CUDA_TRY(cudaMemset(m->d_m, 0, (size_t)m->L.total * 4));
    CUDA_TRY(cudaMemset(m->d_v, 0, (size_t)m->L.total * 4));
    m->step = 0;
    return FFT3_OK;
}

int fft3_mlp_get_params(fft3_mlp m, float *h_params)
{
    if (!m || !h_params)
        return fail(FFT3_ERR_INVALID_ARG, "null argument");
    CUDA_TRY(cudaMemcpy(h_params, m->d_p, (size_t)m->L.total * 4, cudaMemcpyDeviceToHost));
    return FFT3_OK;
}

int fft3_mlp_forward(fft3_mlp m, const float *d_X, int B, float *d_pred, void *stream)
{
    if (!m || !d_X || !d_pred || B < 1)
        return fail(FFT3_ERR_INVALID_ARG, "bad argument to fft3_mlp_forward");
    int rc = mlp_reserve(m, B);
    if (!rc)
        rc = mlp_fwd(m, d_X, B, (cudaStream_t)stream);
    if (rc)
        return rc;
    CUDA_TRY(cudaMemcpyAsync(d_pred, m->z3, (size_t)B * 4, cudaMemcpyDeviceToDevice, (cudaStream_t)stream));
    return FFT3_OK;
}

int fft3_mlp_grad(fft3_mlp m, const float *d_X, const float *d_y, int B, float *d_grad, float *d_loss, void *stream)
{
    if (!m || !d_X || !d_y || B < 1)
        return fail(FFT3_ERR_INVALID_ARG, "bad argument to fft3_mlp_grad");
    cudaStream_t st = (cudaStream_t)stream;
    if (m->grad_ws)
        return mlp_gradient(m, d_X, d_y, nullptr, B, d_grad, d_loss, st);
    int rc = mlp_reserve(m, B);
    if (!rc)
        rc = mlp_fwd(m, d_X, B, st);
    if (!rc)
        rc = mlp_bwd(m, d_X, d_y, B, st);
    if (rc)
        return rc;
    if (d_grad)
        CUDA_TRY(cudaMemcpyAsync(d_grad, m->d_g, (size_t)m->L.total * 4, cudaMemcpyDeviceToDevice, st));
    if (d_loss)
        CUDA_TRY(cudaMemcpyAsync(d_loss, m->loss, 4, cudaMemcpyDeviceToDevice, st));
    return FFT3_OK;
}

int fft3_mlp_adam_step(fft3_mlp m, const float *d_grad, float lr, void *stream)
{
    if (!m || lr <= 0.f)
        return fail(FFT3_ERR_INVALID_ARG, "bad argument to fft3_mlp_adam_step");
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    m->step += 1;
    const float c1 = 1.f - powf(b1, (float)m->step), c2 = 1.f - powf(b2, (float)m->step);
    const float *g = d_grad ? d_grad : m->d_g;
    float b1v = b1, b2v = b2, epsv = eps, c1v = c1, c2v = c2;
    int n = m->L.total;
    void *args[] = {&m->d_p, &g, &m->d_m, &m->d_v, &n, &lr, &b1v, &b2v, &epsv, &c1v, &c2v};
    CUDA_TRY(launch_after((const void *)&k_mlp_adam, nblk(n), 256, 0, (cudaStream_t)stream, args));
    return FFT3_OK;
}

int fft3_mlp_train(fft3_mlp m, const float *h_X, const float *h_y, int n, int epochs, int batch, float lr,
                   unsigned long long seed, float *h_loss_curve)
{
    if (!m || !h_X || !h_y || n < 1 || epochs < 1 || batch < 1 || lr <= 0.f)
        return fail(FFT3_ERR_INVALID_ARG, "bad argument to fft3_mlp_train");
    const int F = m->L.F;
    batch = std::min(batch, n);
    float *dX = nullptr, *dy = nullptr, *dXb = nullptr, *dyb = nullptr;
    int *didx = nullptr;
    auto cleanup = [&]() {
        cudaFree(dX);
        cudaFree(dy);
        cudaFree(dXb);
        cudaFree(dyb);
        cudaFree(didx);
    };
    // gathered minibatches and activations: the layer-by-layer kernels alone need them
    const bool layers = !m->grad_ws;
    if (cudaMalloc(&dX, (size_t)n * F * 4) || cudaMalloc(&dy, (size_t)n * 4) ||
        (layers && (cudaMalloc(&dXb, (size_t)batch * F * 4) || cudaMalloc(&dyb, (size_t)batch * 4))) ||
        cudaMalloc(&didx, (size_t)n * 4)) {
        cudaGetLastError();
        cleanup();
        return fail(FFT3_ERR_OOM, "training buffers");
    }
    cudaMemcpy(dX, h_X, (size_t)n * F * 4, cudaMemcpyHostToDevice);
    cudaMemcpy(dy, h_y, (size_t)n * 4, cudaMemcpyHostToDevice);
    int rc = layers ? mlp_reserve(m, n) : FFT3_OK;
    std::vector<int> perm(n);
    for (int i = 0; i < n; ++i)
        perm[i] = i;
    std::mt19937_64 rng(seed);
    for (int ep = 0; ep < epochs && !rc; ++ep) {
        std::shuffle(perm.begin(), perm.end(), rng);
        cudaMemcpy(didx, perm.data(), (size_t)n * 4, cudaMemcpyHostToDevice);
        for (int s = 0; s < n && !rc; s += batch) {
            const int b = std::min(batch, n - s);
            if (m->grad_ws) {
                rc = mlp_gradient(m, dX, dy, didx + s, b, nullptr, nullptr, nullptr);
            } else {
                k_mlp_gather<<<nblk(b * (F + 1)), 256>>>(dX, dy, didx + s, b, F, dXb, dyb);
                rc = mlp_fwd(m, dXb, b, nullptr);
                if (!rc)
                    rc = mlp_bwd(m, dXb, dyb, b, nullptr);
            }
            if (!rc)
                rc = fft3_mlp_adam_step(m, nullptr, lr, nullptr);
        }
        if (!rc && h_loss_curve) {
            // full-data loss after the epoch
            if (m->grad_ws) {
                rc = mlp_gradient(m, dX, dy, nullptr, n, nullptr, nullptr, nullptr);
            } else {
                rc = mlp_fwd(m, dX, n, nullptr);
                if (!rc)
                    rc = mlp_bwd(m, dX, dy, n, nullptr);
            }
            float l = 0.f;
            if (!rc && cudaMemcpy(&l, m->loss, 4, cudaMemcpyDeviceToHost) != cudaSuccess)
                rc = fail(FFT3_ERR_CUDA, "loss readback");
            h_loss_curve[ep] = l;
        }
    }
    if (!rc && cudaDeviceSynchronize() != cudaSuccess)
        rc = fail(FFT3_ERR_CUDA, "training failed");
    cleanup();
    return rc;
}

int fft3_mlp_predict(fft3_mlp m, const float *h_X, int n, float *h_pred)
{
    if (!m || !h_X || !h_pred || n < 1)
        return fail(FFT3_ERR_INVALID_ARG, "bad argument to fft3_mlp_predict");
    float *dX = nullptr;
    if (cudaMalloc(&dX, (size_t)n * m->L.F * 4)) {
        cudaGetLastError();
        return fail(FFT3_ERR_OOM, "predict buffer");
    }
    cudaMemcpy(dX, h_X, (size_t)n * m->L.F * 4, cudaMemcpyHostToDevice);
    int rc = mlp_reserve(m, n);
    if (!rc)
        rc = mlp_fwd(m, dX, n, nullptr);
    if (!rc && cudaMemcpy(h_pred, m->z3, (size_t)n * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
        rc = fail(FFT3_ERR_CUDA, "predict readback");
    cudaFree(dX);
    return rc;
}

} // extern "C"
