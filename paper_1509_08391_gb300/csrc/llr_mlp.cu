// llr_mlp.cu -- the learned warm start of the Robbins-Monro iteration: a
// 3 -> 64 -> 64 -> 64 -> 1 GELU multilayer perceptron mapping
// (1/V, E/6V, dE/6V), V = L^4, to the slope a, with hand-written FP32
// forward, backward and Adam kernels.  1/V is the volume feature because the
// finite-volume corrections of a_k are O(1/V) (appendix, eq. (A.12)).
//
// The paper's a_k are intrinsic quantities (Sec. 2.2, eq. (2.5); appendix,
// eqs. (A.11)-(A.13)), so a map learned on small volumes can predict the
// slopes of larger ones, and Sec. 2.4 only asks the initial a to be close.
//
// Layout: one float array of parameters, W1 (3x64, row-major [in][out]),
// b1 (64), W2 (64x64), b2, W3 (64x64), b3, W4 (64x1), b4 (1).  Activations
// are [sample][feature].  Layers are small (no tensor cores: a 64-wide layer is
// not a contraction worth them), and the sums over samples are done in a fixed
// order (no atomics), so training is deterministic.  Training runs all its epochs
// in one launch of a cluster of CTAs; predictions and single gradients use a
// thread-per-output kernel per layer.
#include <cmath>
#include <string>
#include <vector>

#include "../../include/llr.h"
#include "llr_internal.h"

namespace {

constexpr int kW = 64;      // hidden width
constexpr int kIn = 3;      // features
constexpr int kNParams = kIn * kW + kW + 2 * (kW * kW + kW) + kW + 1;   // 8641
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kIn * kW, kOffW2 = kOffB1 + kW,
              kOffB2 = kOffW2 + kW * kW, kOffW3 = kOffB2 + kW, kOffB3 = kOffW3 + kW * kW,
              kOffW4 = kOffB3 + kW, kOffB4 = kOffW4 + kW;

__device__ __forceinline__ float gelu(float z)
{
    return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f));
}

__device__ __forceinline__ float gelu_grad(float z)
{
    const float h = 1.0f + erff(z * 0.70710678118654752f), e = z * expf(-0.5f * z * z);
    return fmaf(0.5f, h, __fmul_rn(e, 0.39894228040143268f));
}

// Raw features (1/V, E/6V, dE/6V) standardised with mean / std.
__global__ void features_kernel(int n, const double *L, const double *e, const double *d,
                                const double *mean, const double *std, float *X)
{
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x) {
        const double L2 = L[s] * L[s];
        const double r[3] = {1.0 / (L2 * L2), e[s], d[s]};
        for (int k = 0; k < 3; ++k) X[s * 3 + k] = (float)((r[k] - mean[k]) / std[k]);
    }
}

// Mean and population standard deviation of the raw features (one CTA).
__global__ void feature_stats_kernel(int n, const double *L, const double *e, const double *d,
                                     double *mean, double *std)
{
    __shared__ double red[3][256];
    const int t = threadIdx.x;
    double s1[3] = {0, 0, 0};
    for (int s = t; s < n; s += 256) {
        const double L2 = L[s] * L[s];
        s1[0] += 1.0 / (L2 * L2);
        s1[1] += e[s];
        s1[2] += d[s];
    }
    for (int k = 0; k < 3; ++k) red[k][t] = s1[k];
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (t < o)
            for (int k = 0; k < 3; ++k) red[k][t] += red[k][t + o];
        __syncthreads();
    }
    double m[3];
    for (int k = 0; k < 3; ++k) m[k] = red[k][0] / n;
    __syncthreads();
    double s2[3] = {0, 0, 0};
    for (int s = t; s < n; s += 256) {
        const double L2 = L[s] * L[s];
        const double r[3] = {1.0 / (L2 * L2), e[s], d[s]};
        for (int k = 0; k < 3; ++k) s2[k] += (r[k] - m[k]) * (r[k] - m[k]);
    }
    for (int k = 0; k < 3; ++k) red[k][t] = s2[k];
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (t < o)
            for (int k = 0; k < 3; ++k) red[k][t] += red[k][t + o];
        __syncthreads();
    }
    if (t == 0)
        for (int k = 0; k < 3; ++k) {
            mean[k] = m[k];
            const double sd = sqrt(red[k][0] / n);
            std[k] = sd > 0.0 ? sd : 1.0;
        }
}

// Z[s][j] = b[j] + sum_i H[s][i] W[i][j];  A = gelu(Z) (or Z for the output).
__global__ void linear_fwd_kernel(int n, int in_dim, int out_dim, const float *H, const float *W,
                                  const float *b, float *Z, float *A, int act)
{
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n * out_dim) return;
    const int s = idx / out_dim, j = idx - s * out_dim;
    float z = b[j];
    for (int i = 0; i < in_dim; ++i) z = fmaf(H[s * in_dim + i], W[i * out_dim + j], z);
    Z[idx] = z;
    A[idx] = act ? gelu(z) : z;
}

// dY = 2 (y - t) / n and the loss mean (y - t)^2 (one CTA reduces the loss).
__global__ void loss_grad_kernel(int n, const float *Y, const double *T, float *dY, double *loss)
{
    __shared__ double red[256];
    double acc = 0.0;
    for (int s = threadIdx.x; s < n; s += 256) {
        const double r = (double)Y[s] - T[s];
        dY[s] = (float)(2.0 * r / n);
        acc += r * r;
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0 && loss) *loss = red[0] / n;
}

// dZin[s][i] = (sum_j dZ[s][j] W[i][j]) * gelu'(Zin[s][i]).
__global__ void linear_bwd_data_kernel(int n, int in_dim, int out_dim, const float *dZ,
                                       const float *W, const float *Zin, float *dZin)
{
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n * in_dim) return;
    const int s = idx / in_dim, i = idx - s * in_dim;
    float g = 0.0f;
    for (int j = 0; j < out_dim; ++j) g = fmaf(dZ[s * out_dim + j], W[i * out_dim + j], g);
    dZin[idx] = g * gelu_grad(Zin[idx]);
}

// gW[i][j] = sum_s H[s][i] dZ[s][j]; gb[j] = sum_s dZ[s][j] (thread per output,
// samples summed in order).
__global__ void linear_bwd_weight_kernel(int n, int in_dim, int out_dim, const float *H,
                                         const float *dZ, float *gW, float *gb)
{
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    const int nw = in_dim * out_dim;
    if (idx < nw) {
        const int i = idx / out_dim, j = idx - i * out_dim;
        float g = 0.0f;
        for (int s = 0; s < n; ++s) g = fmaf(H[s * in_dim + i], dZ[s * out_dim + j], g);
        gW[idx] = g;
    } else if (idx < nw + out_dim) {
        const int j = idx - nw;
        float g = 0.0f;
        for (int s = 0; s < n; ++s) g += dZ[s * out_dim + j];
        gb[j] = g;
    }
}

// ---------------------------------------------------------------------------
// Training: all epochs of a fit in one launch of a cluster of kCtas CTAs.
//
// An epoch is two parallel phases with a cluster barrier after each.
//   1. Forward and backward of the samples, which only need the parameters: CTA c
//      takes a contiguous share of the samples, in tiles of kTile, with all
//      parameters in shared memory; activations and dZ go to global memory (L2).
//   2. Parameter gradients and Adam: CTA c owns rows 8 c .. 8 c + 7 of W2 and W3,
//      the first three CTAs the small tensors besides.  A thread keeps its
//      parameters and their moments in registers for the whole training, sums
//      its gradients over all samples (staged through shared memory, kChunk at a
//      time) and writes the new values into every CTA's shared memory.
// Every sum runs over the same terms in the same order as in the kernels above,
// and the fused operations are written out as those round, so results do not
// depend on the split, bit for bit.  Bound by shared-memory loads: four
// samples, or four rows, per thread share a weight or a dZ.  One epoch of 120
// samples took 70 us as 14 launches of a captured graph and takes 12 us here (1000
// samples 262 -> 79 us), the latency of some 15 short dependent steps.
// ---------------------------------------------------------------------------
constexpr int kCtas = 8, kTrainThreads = 512, kTile = 16, kChunk = 128;
constexpr int kRow = kW / kCtas;        // rows of W2, W3 owned by a CTA
constexpr int kWs = kW + 1;             // padded row of a weight matrix
constexpr int kHs = kW + 4;             // padded row of a sample tile (16-byte rows)

struct TrainSmem {
    float W2[kW * kWs], W3[kW * kWs];
    float W1[kIn * kW], b1[kW], b2[kW], b3[kW], W4[kW], b4;
    // phase 1: a tile of samples
    float X[kTile * kIn];
    alignas(16) float H[3][kTile * kHs];    // activations
    alignas(16) float D[3][kTile * kHs];    // gelu'(Z), then dZ
    float dY[kTile];
    // phase 2: a chunk of samples
    alignas(16) float dZ[2][kChunk * kW];   // of layers 2, 3
    alignas(16) float A[2][kChunk * kRow];  // the owned columns of A1, A2
    alignas(16) float E[kChunk * kW];       // CTA 1: dZ1, CTA 2: A3
    float e[kChunk * kIn];                  // CTA 1: X, CTA 2: dY
};

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Store v to the copy of *p in every CTA of the cluster.
__device__ __forceinline__ void store_all(float *p, float v)
{
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
#pragma unroll
    for (int r = 0; r < kCtas; ++r) {
        unsigned d;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(r));
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(d), "f"(v) : "memory");
    }
}

__device__ __forceinline__ void copy16(float *dst, const float *src)   // through L2 only
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}

// Adam (Kingma & Ba 2015) with bias correction, c1, c2 = 1 - b^t.
struct AdamStep {
    float lr, b1, b2, eps, c1, c2;
    __device__ __forceinline__ AdamStep(float lr_, float b1_, float b2_, float eps_, int t)
        : lr(lr_), b1(b1_), b2(b2_), eps(eps_)
    {
        c1 = 1.0f - powf(b1, (float)t);
        c2 = 1.0f - powf(b2, (float)t);
    }
    __device__ __forceinline__ void operator()(float &P, float &M, float &V, float g) const
    {
        M = fmaf(1.0f - b1, g, __fmul_rn(b1, M));
        V = fmaf(__fmul_rn(1.0f - b2, g), g, __fmul_rn(b2, V));
        P -= lr * (M / c1) / (sqrtf(V / c2) + eps);
    }
};

// out[s][j] of a 64 x 64 layer for four samples: sum over i of in[s][i] W(i, j),
// in the order of i, from z.
template <class Weight>
__device__ __forceinline__ void dot4(const float *in, Weight W, float z[4])
{
#pragma unroll
    for (int i = 0; i < kW; i += 4) {
        const float w0 = W(i), w1 = W(i + 1), w2 = W(i + 2), w3 = W(i + 3);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 h = *(const float4 *)(in + q * kHs + i);
            z[q] = fmaf(h.x, w0, z[q]);
            z[q] = fmaf(h.y, w1, z[q]);
            z[q] = fmaf(h.z, w2, z[q]);
            z[q] = fmaf(h.w, w3, z[q]);
        }
    }
}

__global__ void __cluster_dims__(kCtas, 1, 1) __launch_bounds__(kTrainThreads, 1)
    train_kernel(int n, int epochs, const float *X, const double *T, float *A, float *dZ,
                 float *dY, float *P, float *M, float *V, int *t, float lr, float b1, float b2,
                 float eps)
{
    extern __shared__ __align__(16) char smem_raw[];
    TrainSmem &sm = *(TrainSmem *)smem_raw;
    const int tid = threadIdx.x, c = blockIdx.x;
    const size_t layer = (size_t)kW * n;   // A and dZ hold layers 1, 2, 3

    // all parameters into shared memory
    for (int k = tid; k < kW * kW; k += kTrainThreads) {
        sm.W2[(k / kW) * kWs + k % kW] = P[kOffW2 + k];
        sm.W3[(k / kW) * kWs + k % kW] = P[kOffW3 + k];
    }
    for (int k = tid; k < kIn * kW; k += kTrainThreads) sm.W1[k] = P[kOffW1 + k];
    if (tid < kW) {
        sm.b1[tid] = P[kOffB1 + tid];
        sm.b2[tid] = P[kOffB2 + tid];
        sm.b3[tid] = P[kOffB3 + tid];
        sm.W4[tid] = P[kOffW4 + tid];
        if (tid == 0) sm.b4 = P[kOffB4];
    }

    // the parameters this thread owns: nk of them, own[q] in the parameter array
    // and at[q] in shared memory.  Threads 0 .. 255: four rows of a column of W2
    // (m = 0) or W3 (m = 1); the others, in the first three CTAs, the rest.
    const int m = tid >> 7, r4 = 4 * ((tid >> 6) & 1), j = tid & 63, e = tid - 256;
    int nk = 0, first = 0;
    float *at = nullptr;
    if (tid < 256) {
        nk = 4;
        first = (m ? kOffW3 : kOffW2) + (kRow * c + r4) * kW + j;
        at = (m ? sm.W3 : sm.W2) + (kRow * c + r4) * kWs + j;
    } else if (c == 0 && e < 2 * kW) {
        nk = 1;
        first = (e < kW ? kOffB2 : kOffB3 - kW) + e;
        at = e < kW ? sm.b2 + e : sm.b3 + e - kW;
    } else if (c == 1) {
        nk = 1;   // W1, b1 are adjacent
        first = kOffW1 + e;
        at = e < kIn * kW ? sm.W1 + e : sm.b1 + e - kIn * kW;
    } else if (c == 2 && e <= kW) {
        nk = 1;   // W4, b4 are adjacent
        first = kOffW4 + e;
        at = e < kW ? sm.W4 + e : &sm.b4;
    }
    float p[4] = {0, 0, 0, 0}, mom[4] = {0, 0, 0, 0}, var[4] = {0, 0, 0, 0};
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (q < nk) {
            p[q] = P[first + q * kW];
            mom[q] = M[first + q * kW];
            var[q] = V[first + q * kW];
        }
    const int t0 = *t;
    const int share = (n + kCtas - 1) / kCtas, s_end = min(n, (c + 1) * share);
    cluster_sync();   // every CTA of the cluster runs; parameters are loaded

    for (int ep = 0; ep < epochs; ++ep) {
        // ------------------------------------------------ phase 1: the samples
        for (int s0 = c * share; s0 < s_end; s0 += kTile) {
            const int ns = min(kTile, s_end - s0);
            if (tid < kTile * kIn) sm.X[tid] = tid < ns * kIn ? X[(size_t)s0 * kIn + tid] : 0.0f;
            __syncthreads();
            // hidden layers: Z to H, then A = gelu(Z) and gelu'(Z)
#pragma unroll
            for (int l = 0; l < 3; ++l) {
                float *H = sm.H[l];
                if (l == 0) {
                    for (int k = tid; k < kTile * kW; k += kTrainThreads) {
                        const int s = k / kW, o = k % kW;
                        float z = sm.b1[o];
#pragma unroll
                        for (int i = 0; i < kIn; ++i)
                            z = fmaf(sm.X[s * kIn + i], sm.W1[i * kW + o], z);
                        H[s * kHs + o] = z;
                    }
                } else if (tid < 256) {
                    const float *W = (l == 1 ? sm.W2 : sm.W3) + j;
                    const float bias = l == 1 ? sm.b2[j] : sm.b3[j];
                    const int s = 4 * (tid >> 6);
                    float z[4] = {bias, bias, bias, bias};
                    dot4(sm.H[l - 1] + s * kHs, [&](int i) { return W[i * kWs]; }, z);
#pragma unroll
                    for (int q = 0; q < 4; ++q) H[(s + q) * kHs + j] = z[q];
                }
                __syncthreads();
                for (int k = tid; k < kTile * kW; k += kTrainThreads) {
                    const int s = k / kW, o = k % kW;
                    const float z = H[s * kHs + o], a = gelu(z);
                    H[s * kHs + o] = a;
                    sm.D[l][s * kHs + o] = gelu_grad(z);
                    if (s < ns) A[l * layer + (size_t)(s0 + s) * kW + o] = a;
                }
                __syncthreads();
            }
            // output and its gradient 2 (y - t) / n
            if (tid < ns) {
                float y = sm.b4;
#pragma unroll
                for (int i = 0; i < kW; ++i) y = fmaf(sm.H[2][tid * kHs + i], sm.W4[i], y);
                const double r = (double)y - T[s0 + tid];
                const float g = (float)(2.0 * r / n);
                sm.dY[tid] = g;
                dY[s0 + tid] = g;
            } else if (tid < kTile) {
                sm.dY[tid] = 0.0f;
            }
            __syncthreads();
            for (int k = tid; k < kTile * kW; k += kTrainThreads) {
                const int s = k / kW, i = k % kW;
                const float g = fmaf(sm.dY[s], sm.W4[i], 0.0f) * sm.D[2][s * kHs + i];
                sm.D[2][s * kHs + i] = g;
                if (s < ns) dZ[2 * layer + (size_t)(s0 + s) * kW + i] = g;
            }
            __syncthreads();
#pragma unroll
            for (int l = 1; l >= 0; --l) {
                if (tid < 256) {
                    const float *W = (l == 1 ? sm.W3 : sm.W2) + j * kWs;
                    const int s = 4 * (tid >> 6);
                    float g[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                    dot4(sm.D[l + 1] + s * kHs, [&](int o) { return W[o]; }, g);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const float d = g[q] * sm.D[l][(s + q) * kHs + j];
                        sm.D[l][(s + q) * kHs + j] = d;
                        if (s + q < ns) dZ[l * layer + (size_t)(s0 + s + q) * kW + j] = d;
                    }
                }
                __syncthreads();
            }
        }
        cluster_sync();
        // ------------------------------------- phase 2: gradients and parameters
        float g[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        for (int c0 = 0; c0 < n; c0 += kChunk) {
            const int nc = min(kChunk, n - c0);
            for (int k = tid; k < nc * (kW / 4); k += kTrainThreads) {
                copy16(sm.dZ[0] + 4 * k, dZ + layer + (size_t)c0 * kW + 4 * k);
                copy16(sm.dZ[1] + 4 * k, dZ + 2 * layer + (size_t)c0 * kW + 4 * k);
                if (c == 1) copy16(sm.E + 4 * k, dZ + (size_t)c0 * kW + 4 * k);
                if (c == 2) copy16(sm.E + 4 * k, A + 2 * layer + (size_t)c0 * kW + 4 * k);
            }
            for (int k = tid; k < nc * (kRow / 4); k += kTrainThreads) {
                const int s = k / (kRow / 4), q = 4 * (k % (kRow / 4));
                const size_t src = (size_t)(c0 + s) * kW + kRow * c + q;
                copy16(sm.A[0] + s * kRow + q, A + src);
                copy16(sm.A[1] + s * kRow + q, A + layer + src);
            }
            if (c == 1)
                for (int k = tid; k < nc * kIn; k += kTrainThreads)
                    sm.e[k] = X[(size_t)c0 * kIn + k];
            if (c == 2)
                for (int k = tid; k < nc; k += kTrainThreads) sm.e[k] = __ldcg(dY + c0 + k);
            asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
            __syncthreads();
            if (tid < 256) {
                const float *dz = sm.dZ[m] + j, *a = sm.A[m] + r4;
#pragma unroll 8
                for (int s = 0; s < nc; ++s) {
                    const float d = dz[s * kW];
                    const float4 h = *(const float4 *)(a + s * kRow);
                    g[0] = fmaf(h.x, d, g[0]);
                    g[1] = fmaf(h.y, d, g[1]);
                    g[2] = fmaf(h.z, d, g[2]);
                    g[3] = fmaf(h.w, d, g[3]);
                }
            } else if (nk) {
                if (c == 0) {
                    const float *dz = sm.dZ[e >> 6] + (e & 63);
#pragma unroll 8
                    for (int s = 0; s < nc; ++s) g[0] += dz[s * kW];
                } else if (c == 1) {
                    const float *dz = sm.E + (e & 63);
                    const int i = e >> 6;   // input of W1, kIn: the bias
                    if (i < kIn) {
#pragma unroll 8
                        for (int s = 0; s < nc; ++s)
                            g[0] = fmaf(sm.e[s * kIn + i], dz[s * kW], g[0]);
                    } else {
#pragma unroll 8
                        for (int s = 0; s < nc; ++s) g[0] += dz[s * kW];
                    }
                } else if (e < kW) {
#pragma unroll 8
                    for (int s = 0; s < nc; ++s) g[0] = fmaf(sm.E[s * kW + e], sm.e[s], g[0]);
                } else {
#pragma unroll 8
                    for (int s = 0; s < nc; ++s) g[0] += sm.e[s];
                }
            }
            __syncthreads();
        }
        const AdamStep adam(lr, b1, b2, eps, t0 + ep + 1);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (q < nk) {
                adam(p[q], mom[q], var[q], g[q]);
                store_all(at + q * kWs, p[q]);
            }
        cluster_sync();
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (q < nk) {
            P[first + q * kW] = p[q];
            M[first + q * kW] = mom[q];
            V[first + q * kW] = var[q];
        }
    if (c == 0 && tid == 0) *t = t0 + epochs;
}

__global__ void to_double_kernel(int n, const float *a, double *b)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) b[k] = (double)a[k];
}

// Initial weights: normal(0, 1/sqrt(fan_in)) from Philox (Box-Muller), zero biases.
__global__ void init_params_kernel(float *P, uint32_t k0, uint32_t k1)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= kNParams) return;
    int fan = 0;
    if (k < kOffB1) fan = kIn;
    else if (k >= kOffW2 && k < kOffB2) fan = kW;
    else if (k >= kOffW3 && k < kOffB3) fan = kW;
    else if (k >= kOffW4 && k < kOffB4) fan = kW;
    if (fan == 0) {
        P[k] = 0.0f;
        return;
    }
    const llr::U4 w = llr::philox4x32_10((uint32_t)k, 0u, 0x4D4Cu, 0u, k0, k1);
    const float u1 = llr::u01(w.x), u2 = llr::u01(w.y);
    const float z = sqrtf(-2.0f * logf(u1)) * cospif(2.0f * u2);
    P[k] = z / sqrtf((float)fan);
}

struct Buffers {
    int n = 0;
    float *X = nullptr, *Z = nullptr, *A = nullptr, *dZ = nullptr, *Y = nullptr, *dY = nullptr;
    double *T = nullptr, *raw = nullptr, *loss = nullptr;
};

}  // namespace

struct llr_mlp {
    cudaStream_t stream = nullptr;
    float *P = nullptr, *G = nullptr, *M = nullptr, *V = nullptr;
    int *t = nullptr;
    double *norm = nullptr;   // mean[3], std[3]
    Buffers buf;
};

namespace {

int fail(int code, const std::string &msg)
{
    return llr::set_last_error(code, msg.c_str());
}

#define MLP_CUDA(call)                                                                     \
    do {                                                                                   \
        cudaError_t e_ = (call);                                                           \
        if (e_ != cudaSuccess)                                                             \
            return fail(LLR_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

unsigned blocks(long long n, int t = 256)
{
    return (unsigned)((n + t - 1) / t);
}

int ensure_buffers(llr_mlp *h, int n)
{
    if (h->buf.n >= n) return LLR_OK;
    Buffers &b = h->buf;
    cudaFree(b.X); cudaFree(b.Z); cudaFree(b.A); cudaFree(b.dZ); cudaFree(b.Y); cudaFree(b.dY);
    cudaFree(b.T); cudaFree(b.raw); cudaFree(b.loss);
    b = Buffers();
    MLP_CUDA(cudaMalloc(&b.X, sizeof(float) * 3 * (size_t)n));
    MLP_CUDA(cudaMalloc(&b.Z, sizeof(float) * 3 * kW * (size_t)n));
    MLP_CUDA(cudaMalloc(&b.A, sizeof(float) * 3 * kW * (size_t)n));
    MLP_CUDA(cudaMalloc(&b.dZ, sizeof(float) * 3 * kW * (size_t)n));
    MLP_CUDA(cudaMalloc(&b.Y, sizeof(float) * (size_t)n));
    MLP_CUDA(cudaMalloc(&b.dY, sizeof(float) * (size_t)n));
    MLP_CUDA(cudaMalloc(&b.T, sizeof(double) * (size_t)n));
    MLP_CUDA(cudaMalloc(&b.raw, sizeof(double) * 4 * (size_t)n));
    MLP_CUDA(cudaMalloc(&b.loss, sizeof(double)));
    b.n = n;
    return LLR_OK;
}

int upload_inputs(llr_mlp *h, int n, const double *L, const double *e, const double *d)
{
    double *r = h->buf.raw;
    MLP_CUDA(cudaMemcpyAsync(r, L, sizeof(double) * n, cudaMemcpyHostToDevice, h->stream));
    MLP_CUDA(cudaMemcpyAsync(r + n, e, sizeof(double) * n, cudaMemcpyHostToDevice, h->stream));
    MLP_CUDA(cudaMemcpyAsync(r + 2 * n, d, sizeof(double) * n, cudaMemcpyHostToDevice,
                             h->stream));
    return LLR_OK;
}

void enqueue_features(llr_mlp *h, int n)
{
    const double *r = h->buf.raw;
    features_kernel<<<blocks(n), 256, 0, h->stream>>>(n, r, r + n, r + 2 * n, h->norm,
                                                      h->norm + 3, h->buf.X);
}

// Forward pass on the standardised features in buf.X; output in buf.Y.
void enqueue_forward(llr_mlp *h, int n)
{
    Buffers &b = h->buf;
    const size_t L1 = 0, L2 = (size_t)kW * n, L3 = 2 * (size_t)kW * n;
    linear_fwd_kernel<<<blocks((long long)n * kW), 256, 0, h->stream>>>(
        n, kIn, kW, b.X, h->P + kOffW1, h->P + kOffB1, b.Z + L1, b.A + L1, 1);
    linear_fwd_kernel<<<blocks((long long)n * kW), 256, 0, h->stream>>>(
        n, kW, kW, b.A + L1, h->P + kOffW2, h->P + kOffB2, b.Z + L2, b.A + L2, 1);
    linear_fwd_kernel<<<blocks((long long)n * kW), 256, 0, h->stream>>>(
        n, kW, kW, b.A + L2, h->P + kOffW3, h->P + kOffB3, b.Z + L3, b.A + L3, 1);
    linear_fwd_kernel<<<blocks(n), 256, 0, h->stream>>>(n, kW, 1, b.A + L3, h->P + kOffW4,
                                                       h->P + kOffB4, b.dY, b.Y, 0);
}

// Loss, gradients into h->G (forward must have run).
void enqueue_backward(llr_mlp *h, int n)
{
    Buffers &b = h->buf;
    const size_t L1 = 0, L2 = (size_t)kW * n, L3 = 2 * (size_t)kW * n;
    loss_grad_kernel<<<1, 256, 0, h->stream>>>(n, b.Y, b.T, b.dY, b.loss);
    linear_bwd_weight_kernel<<<blocks(kW + 1), 256, 0, h->stream>>>(
        n, kW, 1, b.A + L3, b.dY, h->G + kOffW4, h->G + kOffB4);
    linear_bwd_data_kernel<<<blocks((long long)n * kW), 256, 0, h->stream>>>(
        n, kW, 1, b.dY, h->P + kOffW4, b.Z + L3, b.dZ + L3);
    linear_bwd_weight_kernel<<<blocks(kW * kW + kW), 256, 0, h->stream>>>(
        n, kW, kW, b.A + L2, b.dZ + L3, h->G + kOffW3, h->G + kOffB3);
    linear_bwd_data_kernel<<<blocks((long long)n * kW), 256, 0, h->stream>>>(
        n, kW, kW, b.dZ + L3, h->P + kOffW3, b.Z + L2, b.dZ + L2);
    linear_bwd_weight_kernel<<<blocks(kW * kW + kW), 256, 0, h->stream>>>(
        n, kW, kW, b.A + L1, b.dZ + L2, h->G + kOffW2, h->G + kOffB2);
    linear_bwd_data_kernel<<<blocks((long long)n * kW), 256, 0, h->stream>>>(
        n, kW, kW, b.dZ + L2, h->P + kOffW2, b.Z + L1, b.dZ + L1);
    linear_bwd_weight_kernel<<<blocks(kIn * kW + kW), 256, 0, h->stream>>>(
        n, kIn, kW, b.X, b.dZ + L1, h->G + kOffW1, h->G + kOffB1);
}

}  // namespace

extern "C" {

int llr_mlp_create(llr_mlp_handle *out, uint64_t seed, void *cuda_stream)
{
    if (!out) return fail(LLR_ERR_ARG, "null handle pointer");
    *out = nullptr;
    llr_mlp *h = new llr_mlp();
    h->stream = (cudaStream_t)cuda_stream;
    *out = h;
    MLP_CUDA(cudaMalloc(&h->P, sizeof(float) * kNParams));
    MLP_CUDA(cudaMalloc(&h->G, sizeof(float) * kNParams));
    MLP_CUDA(cudaMalloc(&h->M, sizeof(float) * kNParams));
    MLP_CUDA(cudaMalloc(&h->V, sizeof(float) * kNParams));
    MLP_CUDA(cudaMalloc(&h->t, sizeof(int)));
    MLP_CUDA(cudaMalloc(&h->norm, sizeof(double) * 6));
    MLP_CUDA(cudaMemsetAsync(h->G, 0, sizeof(float) * kNParams, h->stream));
    MLP_CUDA(cudaMemsetAsync(h->M, 0, sizeof(float) * kNParams, h->stream));
    MLP_CUDA(cudaMemsetAsync(h->V, 0, sizeof(float) * kNParams, h->stream));
    MLP_CUDA(cudaMemsetAsync(h->t, 0, sizeof(int), h->stream));
    const double init_norm[6] = {0, 0, 0, 1, 1, 1};
    MLP_CUDA(cudaMemcpy(h->norm, init_norm, sizeof(init_norm), cudaMemcpyHostToDevice));
    init_params_kernel<<<blocks(kNParams), 256, 0, h->stream>>>(h->P, (uint32_t)seed,
                                                                (uint32_t)(seed >> 32));
    MLP_CUDA(cudaGetLastError());
    MLP_CUDA(cudaStreamSynchronize(h->stream));
    return LLR_OK;
}

int llr_mlp_num_params(void)
{
    return kNParams;
}

int llr_mlp_get_params(llr_mlp_handle h, float *out)
{
    if (!h || !out) return fail(LLR_ERR_ARG, "null argument");
    MLP_CUDA(cudaMemcpyAsync(out, h->P, sizeof(float) * kNParams, cudaMemcpyDeviceToHost,
                             h->stream));
    MLP_CUDA(cudaStreamSynchronize(h->stream));
    return LLR_OK;
}

int llr_mlp_set_params(llr_mlp_handle h, const float *in)
{
    if (!h || !in) return fail(LLR_ERR_ARG, "null argument");
    MLP_CUDA(cudaMemcpyAsync(h->P, in, sizeof(float) * kNParams, cudaMemcpyHostToDevice,
                             h->stream));
    MLP_CUDA(cudaMemsetAsync(h->M, 0, sizeof(float) * kNParams, h->stream));
    MLP_CUDA(cudaMemsetAsync(h->V, 0, sizeof(float) * kNParams, h->stream));
    MLP_CUDA(cudaMemsetAsync(h->t, 0, sizeof(int), h->stream));
    MLP_CUDA(cudaStreamSynchronize(h->stream));
    return LLR_OK;
}

int llr_mlp_set_norm(llr_mlp_handle h, const double *mean, const double *std)
{
    if (!h || !mean || !std) return fail(LLR_ERR_ARG, "null argument");
    for (int k = 0; k < 3; ++k)
        if (!(std[k] > 0.0) || !std::isfinite(mean[k]))
            return fail(LLR_ERR_ARG, "std must be positive and mean finite");
    const double v[6] = {mean[0], mean[1], mean[2], std[0], std[1], std[2]};
    MLP_CUDA(cudaMemcpyAsync(h->norm, v, sizeof(v), cudaMemcpyHostToDevice, h->stream));
    MLP_CUDA(cudaStreamSynchronize(h->stream));
    return LLR_OK;
}

int llr_mlp_get_norm(llr_mlp_handle h, double *mean, double *std)
{
    if (!h || !mean || !std) return fail(LLR_ERR_ARG, "null argument");
    double v[6];
    MLP_CUDA(cudaMemcpyAsync(v, h->norm, sizeof(v), cudaMemcpyDeviceToHost, h->stream));
    MLP_CUDA(cudaStreamSynchronize(h->stream));
    for (int k = 0; k < 3; ++k) {
        mean[k] = v[k];
        std[k] = v[3 + k];
    }
    return LLR_OK;
}

static int check_inputs(int n, const double *L, const double *e, const double *d)
{
    if (n < 1 || !L || !e || !d) return fail(LLR_ERR_ARG, "need n >= 1 and input arrays");
    for (int s = 0; s < n; ++s)
        if (!(L[s] > 0.0) || !std::isfinite(e[s]) || !std::isfinite(d[s]))
            return fail(LLR_ERR_ARG, "inputs must be finite with L > 0");
    return LLR_OK;
}

int llr_mlp_predict(llr_mlp_handle h, int n, const double *L, const double *e6v,
                    const double *dE6v, double *a_out)
{
    if (!h || !a_out) return fail(LLR_ERR_ARG, "null argument");
    if (int r = check_inputs(n, L, e6v, dE6v)) return r;
    if (int r = ensure_buffers(h, n)) return r;
    if (int r = upload_inputs(h, n, L, e6v, dE6v)) return r;
    enqueue_features(h, n);
    enqueue_forward(h, n);
    to_double_kernel<<<blocks(n), 256, 0, h->stream>>>(n, h->buf.Y, h->buf.T);
    MLP_CUDA(cudaGetLastError());
    MLP_CUDA(cudaMemcpyAsync(a_out, h->buf.T, sizeof(double) * n, cudaMemcpyDeviceToHost,
                             h->stream));
    MLP_CUDA(cudaStreamSynchronize(h->stream));
    return LLR_OK;
}

int llr_mlp_grad(llr_mlp_handle h, int n, const double *L, const double *e6v,
                 const double *dE6v, const double *a_target, float *grad_out, double *loss_out)
{
    if (!h || !a_target || !grad_out) return fail(LLR_ERR_ARG, "null argument");
    if (int r = check_inputs(n, L, e6v, dE6v)) return r;
    if (int r = ensure_buffers(h, n)) return r;
    if (int r = upload_inputs(h, n, L, e6v, dE6v)) return r;
    MLP_CUDA(cudaMemcpyAsync(h->buf.T, a_target, sizeof(double) * n, cudaMemcpyHostToDevice,
                             h->stream));
    enqueue_features(h, n);
    enqueue_forward(h, n);
    enqueue_backward(h, n);
    MLP_CUDA(cudaGetLastError());
    MLP_CUDA(cudaMemcpyAsync(grad_out, h->G, sizeof(float) * kNParams, cudaMemcpyDeviceToHost,
                             h->stream));
    double loss = 0.0;
    MLP_CUDA(cudaMemcpyAsync(&loss, h->buf.loss, sizeof(double), cudaMemcpyDeviceToHost,
                             h->stream));
    MLP_CUDA(cudaStreamSynchronize(h->stream));
    if (loss_out) *loss_out = loss;
    return LLR_OK;
}

int llr_mlp_fit(llr_mlp_handle h, int n, const double *L, const double *e6v, const double *dE6v,
                const double *a_target, int epochs, double lr, int standardise,
                double *loss_out)
{
    if (!h || !a_target) return fail(LLR_ERR_ARG, "null argument");
    if (epochs < 0 || !(lr > 0.0)) return fail(LLR_ERR_ARG, "epochs >= 0 and lr > 0");
    if (int r = check_inputs(n, L, e6v, dE6v)) return r;
    if (int r = ensure_buffers(h, n)) return r;
    if (int r = upload_inputs(h, n, L, e6v, dE6v)) return r;
    MLP_CUDA(cudaMemcpyAsync(h->buf.T, a_target, sizeof(double) * n, cudaMemcpyHostToDevice,
                             h->stream));
    const double *r = h->buf.raw;
    if (standardise)
        feature_stats_kernel<<<1, 256, 0, h->stream>>>(n, r, r + n, r + 2 * n, h->norm,
                                                       h->norm + 3);
    enqueue_features(h, n);
    MLP_CUDA(cudaGetLastError());
    if (epochs > 0) {
        Buffers &b = h->buf;
        MLP_CUDA(cudaFuncSetAttribute(train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)sizeof(TrainSmem)));
        train_kernel<<<kCtas, kTrainThreads, sizeof(TrainSmem), h->stream>>>(
            n, epochs, b.X, b.T, b.A, b.dZ, b.dY, h->P, h->M, h->V, h->t, (float)lr,
            0.9f, 0.999f, 1e-8f);
        MLP_CUDA(cudaGetLastError());
    }
    // loss of the final parameters
    enqueue_forward(h, n);
    loss_grad_kernel<<<1, 256, 0, h->stream>>>(n, h->buf.Y, h->buf.T, h->buf.dY, h->buf.loss);
    MLP_CUDA(cudaGetLastError());
    double loss = 0.0;
    MLP_CUDA(cudaMemcpyAsync(&loss, h->buf.loss, sizeof(double), cudaMemcpyDeviceToHost,
                             h->stream));
    MLP_CUDA(cudaStreamSynchronize(h->stream));
    if (loss_out) *loss_out = loss;
    return LLR_OK;
}

int llr_mlp_destroy(llr_mlp_handle h)
{
    if (!h) return LLR_OK;
    if (h->stream) cudaStreamSynchronize(h->stream);
    else cudaDeviceSynchronize();
    Buffers &b = h->buf;
    cudaFree(b.X); cudaFree(b.Z); cudaFree(b.A); cudaFree(b.dZ); cudaFree(b.Y); cudaFree(b.dY);
    cudaFree(b.T); cudaFree(b.raw); cudaFree(b.loss);
    cudaFree(h->P); cudaFree(h->G); cudaFree(h->M); cudaFree(h->V); cudaFree(h->t);
    cudaFree(h->norm);
    delete h;
    return LLR_OK;
}

}  // extern "C"
