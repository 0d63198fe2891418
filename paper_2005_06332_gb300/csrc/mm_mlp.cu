// mm_mlp.cu -- the learned cost model: a 16 -> 64 -> 64 -> 1 MLP (ReLU),
// BF16 weights, FP32 accumulation, trained with Adam on FP32 master
// weights, by hand-written kernels.
//
// It predicts a neuron's per-step solve time from its morphology features
// so that the work queue can take the longest items first (the paper's
// priority(size) and sorting by size, Sec. 4, with a learned key).
//
// Parameters, flat, in this order (MM_MLP_PARAMS = 5313 values):
//   W1 [64 x 16] row-major, b1 [64], W2 [64 x 64], b2 [64], W3 [1 x 64], b3 [1].
// Inputs are standardised with per-feature mean / std, targets with mean /
// std, both taken from the training set by mm_mlp_train.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>
#include <cstring>
#include <new>
#include <random>
#include <type_traits>
#include <vector>

#include "mm.h"

namespace {

constexpr int kIn = MM_N_FEATURES, kH = 64;
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kH * kIn, kOffW2 = kOffB1 + kH, kOffB2 = kOffW2 + kH * kH,
              kOffW3 = kOffB2 + kH, kOffB3 = kOffW3 + kH, kParams = kOffB3 + 1;
static_assert(kParams == MM_MLP_PARAMS, "parameter count");

// The parameters and the standardisation, as the kernels take them.
struct Model {
    const __nv_bfloat16 *w;
    const float *mu, *sd;
    float y_mu, y_sd;
};

__device__ __forceinline__ float weight(const Model &m, int i) { return __bfloat162float(m.w[i]); }

// Forward, two samples per thread: the first hidden layer stays in registers,
// the weights (widened to FP32, transposed so that the weights of eight units
// of one input are two 16-byte reads) in shared memory, where all lanes read
// the same one.  Bound by the registers' side of shared memory (a 16-byte read
// of a warp takes four clocks), hence two samples for each read, and by FP32
// issue (5,184 multiply-adds a sample).  100,000 samples: 1.53 ms with a thread
// per (sample, unit) of each layer, whose lanes read weights 128 bytes apart;
// 0.070 ms with one sample per thread, 0.054 ms with two.
constexpr int kFwdThreads = 128, kFwdSamples = 2;

__global__ void __launch_bounds__(kFwdThreads) predict_kernel(Model m, const float *__restrict__ X, int64_t n,
                                                              float *__restrict__ out)
{
    __shared__ __align__(16) float w1[kIn * kH], w2[kH * kH];
    __shared__ float b1[kH], b2[kH], w3[kH], mu[kIn], sd[kIn];
    for (int i = threadIdx.x; i < kH * kH; i += kFwdThreads) w2[(i % kH) * kH + i / kH] = weight(m, kOffW2 + i);
    for (int i = threadIdx.x; i < kH * kIn; i += kFwdThreads) w1[(i % kIn) * kH + i / kIn] = weight(m, kOffW1 + i);
    for (int i = threadIdx.x; i < kH; i += kFwdThreads) {
        b1[i] = weight(m, kOffB1 + i);
        b2[i] = weight(m, kOffB2 + i);
        w3[i] = weight(m, kOffW3 + i);
        if (i < kIn) {
            mu[i] = m.mu[i];
            sd[i] = m.sd[i];
        }
    }
    const float b3 = weight(m, kOffB3);
    __syncthreads();
    // eight units u .. u+7 of the samples: b[u] + sum_k in[k] w[k][u], k ascending
    auto units = [&](const float *w, const float *b, int u, auto K, const auto &in, float acc[kFwdSamples][8]) {
#pragma unroll
        for (int q = 0; q < kFwdSamples; ++q)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[q][j] = b[u + j];
#pragma unroll
        for (int k = 0; k < decltype(K)::value; ++k) {
            const float4 f = *(const float4 *)(w + k * kH + u), g = *(const float4 *)(w + k * kH + u + 4);
            const float wv[8] = {f.x, f.y, f.z, f.w, g.x, g.y, g.z, g.w};
#pragma unroll
            for (int q = 0; q < kFwdSamples; ++q)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[q][j] = fmaf(in[q][k], wv[j], acc[q][j]);
        }
    };
    constexpr int kStep = kFwdThreads * kFwdSamples;
    for (int64_t s0 = blockIdx.x * (int64_t)kStep + threadIdx.x; s0 < n; s0 += (int64_t)gridDim.x * kStep) {
        asm volatile("" ::: "memory");  // the weights are read again for each sample, not kept (and spilled)
        float x[kFwdSamples][kIn], h[kFwdSamples][kH], acc[kFwdSamples][8], y[kFwdSamples];
#pragma unroll
        for (int q = 0; q < kFwdSamples; ++q) {
            const int64_t s = s0 + q * kFwdThreads < n ? s0 + q * kFwdThreads : n - 1;
#pragma unroll
            for (int k = 0; k < kIn; k += 4) {
                const float4 v = ((const float4 *)X)[s * (kIn / 4) + k / 4];
                x[q][k] = (v.x - mu[k]) / sd[k];
                x[q][k + 1] = (v.y - mu[k + 1]) / sd[k + 1];
                x[q][k + 2] = (v.z - mu[k + 2]) / sd[k + 2];
                x[q][k + 3] = (v.w - mu[k + 3]) / sd[k + 3];
            }
            y[q] = b3;
        }
#pragma unroll
        for (int u = 0; u < kH; u += 8) {
            units(w1, b1, u, std::integral_constant<int, kIn>{}, x, acc);
#pragma unroll
            for (int q = 0; q < kFwdSamples; ++q)
#pragma unroll
                for (int j = 0; j < 8; ++j) h[q][u + j] = fmaxf(acc[q][j], 0.0f);
        }
#pragma unroll 1
        for (int u = 0; u < kH; u += 8) {
            units(w2, b2, u, std::integral_constant<int, kH>{}, h, acc);
#pragma unroll
            for (int q = 0; q < kFwdSamples; ++q)
#pragma unroll
                for (int j = 0; j < 8; ++j) y[q] = fmaf(fmaxf(acc[q][j], 0.0f), w3[u + j], y[q]);
        }
#pragma unroll
        for (int q = 0; q < kFwdSamples; ++q)
            if (s0 + q * kFwdThreads < n) out[s0 + q * kFwdThreads] = fmaf(y[q], m.y_sd, m.y_mu);
    }
}

// Loss and gradient of tiles of kTile samples: forward, the mean squared
// error's derivative, and the gradients of the layers, with everything of a
// tile in shared memory.  A lane holds a sample and a warp eight units of a
// layer; for the weights' gradients a thread holds 4 x 4 of W2's and four of
// W1's, which it sums over the block's tiles in registers.  Each block leaves
// its sums in part[block * kPart ...] (the loss last), added in block order by
// sum_kernel: the same result every time.  5,000 samples: forward and backward
// 1.6 ms with a thread per weight that walks all samples (23 blocks busy),
// 0.031 ms so (0.025 ms here, 0.006 ms in sum_kernel), and the gradient's error
// against FP64 7e-7 -> 6e-8 (shorter sums).
constexpr int kTile = 32, kGradThreads = 256, kRow = kTile + 4;  // row stride: 16-byte reads of eight rows without conflicts
constexpr int kPart = kParams + 1;
constexpr int kMaxPart = 304;  // two blocks per SM

struct GradSmem {
    float w1[kIn * kH];              // [k][u]
    float w2t[kH * kH];              // [k][u]
    float w2[kH * kH];               // [u][k]
    float x[kIn * kRow], h1[kH * kRow], g2[kH * kRow], g1[kH * kRow];  // [unit][sample]; g2: h2, then its gradient
    float b1[kH], b2[kH], w3[kH], dy[kTile], y[kTile];
};

__global__ void __launch_bounds__(kGradThreads, 2) loss_grad_kernel(Model m, const float *__restrict__ X,
                                                                 const float *__restrict__ Y, int64_t n,
                                                                 float *__restrict__ part)
{
    extern __shared__ __align__(16) unsigned char raw[];
    GradSmem &S = *(GradSmem *)raw;
    const int tid = threadIdx.x, lane = tid & 31, u0 = (tid >> 5) * 8;
    for (int i = tid; i < kH * kH; i += kGradThreads) {
        const float w = weight(m, kOffW2 + i);
        S.w2[i] = w;
        S.w2t[(i % kH) * kH + i / kH] = w;
    }
    for (int i = tid; i < kH * kIn; i += kGradThreads) S.w1[(i % kIn) * kH + i / kIn] = weight(m, kOffW1 + i);
    if (tid < kH) {
        S.b1[tid] = weight(m, kOffB1 + tid);
        S.b2[tid] = weight(m, kOffB2 + tid);
        S.w3[tid] = weight(m, kOffW3 + tid);
    }
    const float b3 = weight(m, kOffB3);
    const int gu = (tid >> 4) * 4, gk = (tid & 15) * 4;  // this thread's 4 x 4 of W2, and W1[gu .. gu+3][tid & 15]
    float a2[4][4] = {}, a1[4] = {}, ab = 0.0f, a3 = 0.0f, loss = 0.0f;  // ab: b1 (tid < 64), b2 (< 128), b3 (128)
    // eight units u0 .. u0+7 of sample `lane`: sum_k in[k][lane] w[k][u], k ascending
    auto layer = [&](const float *in, const float *w, int K, float acc[8]) {
#pragma unroll 8
        for (int k = 0; k < K; ++k) {
            const float4 p = *(const float4 *)(w + k * kH + u0), q = *(const float4 *)(w + k * kH + u0 + 4);
            const float v = in[k * kRow + lane];
            const float wv[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[j] = fmaf(v, wv[j], acc[j]);
        }
    };
    for (int64_t t = blockIdx.x; t * kTile < n; t += gridDim.x) {
        __syncthreads();
        for (int i = tid; i < kTile * kIn; i += kGradThreads) {
            const int64_t s = t * kTile + i / kIn;
            const int k = i % kIn;
            S.x[k * kRow + i / kIn] = s < n ? (X[s * kIn + k] - m.mu[k]) / m.sd[k] : 0.0f;
        }
        __syncthreads();
        float acc[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j] = S.b1[u0 + j];
        layer(S.x, S.w1, kIn, acc);
#pragma unroll
        for (int j = 0; j < 8; ++j) S.h1[(u0 + j) * kRow + lane] = fmaxf(acc[j], 0.0f);
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j] = S.b2[u0 + j];
        layer(S.h1, S.w2t, kH, acc);
#pragma unroll
        for (int j = 0; j < 8; ++j) S.g2[(u0 + j) * kRow + lane] = fmaxf(acc[j], 0.0f);
        __syncthreads();
        if (tid < kTile) {
            float y = b3;
            for (int k = 0; k < kH; ++k) y = fmaf(S.g2[k * kRow + tid], S.w3[k], y);
            const int64_t s = t * kTile + tid;
            const float e = s < n ? y - (Y[s] - m.y_mu) / m.y_sd : 0.0f;
            S.dy[tid] = 2.0f * e / (float)n;
            loss = fmaf(e, e, loss);
        }
        __syncthreads();
        // W3 and b3, then h2's gradient in h2's place
        if (tid < kH) {
            for (int s = 0; s < kTile; ++s) a3 = fmaf(S.dy[s], S.g2[tid * kRow + s], a3);
        } else if (tid == 128) {
            for (int s = 0; s < kTile; ++s) ab += S.dy[s];
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            float *h = &S.g2[(u0 + j) * kRow + lane];
            *h = *h > 0.0f ? S.dy[lane] * S.w3[u0 + j] : 0.0f;
        }
        __syncthreads();
        // h1's gradient: sum_u g2[u] W2[u][k], the roles of u and k exchanged
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j] = 0.0f;
        layer(S.g2, S.w2, kH, acc);
#pragma unroll
        for (int j = 0; j < 8; ++j)
            S.g1[(u0 + j) * kRow + lane] = S.h1[(u0 + j) * kRow + lane] > 0.0f ? acc[j] : 0.0f;
        __syncthreads();
#pragma unroll 2
        for (int s = 0; s < kTile; s += 4) {
            float4 g[4], h[4], d[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                g[j] = *(const float4 *)&S.g2[(gu + j) * kRow + s];
                h[j] = *(const float4 *)&S.h1[(gk + j) * kRow + s];
                d[j] = *(const float4 *)&S.g1[(gu + j) * kRow + s];
            }
            const float4 xv = *(const float4 *)&S.x[(tid & 15) * kRow + s];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    a2[i][j] = fmaf(g[i].w, h[j].w, fmaf(g[i].z, h[j].z, fmaf(g[i].y, h[j].y, fmaf(g[i].x, h[j].x, a2[i][j]))));
                a1[i] = fmaf(d[i].w, xv.w, fmaf(d[i].z, xv.z, fmaf(d[i].y, xv.y, fmaf(d[i].x, xv.x, a1[i]))));
            }
        }
        if (tid < 128) {
            const float *g = tid < kH ? &S.g1[tid * kRow] : &S.g2[(tid - kH) * kRow];
            for (int s = 0; s < kTile; ++s) ab += g[s];
        }
    }
    float *P = part + (int64_t)blockIdx.x * kPart;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
        for (int j = 0; j < 4; ++j) P[kOffW2 + (gu + i) * kH + gk + j] = a2[i][j];
        P[kOffW1 + (gu + i) * kIn + (tid & 15)] = a1[i];
    }
    if (tid < kH) {
        P[kOffB1 + tid] = ab;
        P[kOffW3 + tid] = a3;
    } else if (tid < 128) {
        P[kOffB2 + tid - kH] = ab;
    } else if (tid == 128) {
        P[kOffB3] = ab;
    }
    if (tid < 32) {
        for (int o = 16; o > 0; o >>= 1) loss += __shfl_down_sync(0xFFFFFFFFu, loss, o);
        if (tid == 0) P[kParams] = loss / (float)n;
    }
}

struct AdamArgs {
    float *w, *m, *v;  // w == nullptr: no step
    __nv_bfloat16 *wb;
    float lr, b1, b2, eps, c1, c2;
};

// The blocks' sums added in block order (eight runs of blocks, then these in
// order): the gradient and the loss, and, when asked for, Adam on the FP32
// master weights, which refreshes the BF16 compute copy.
__global__ void __launch_bounds__(256) sum_kernel(const float *__restrict__ part, int blocks, float *__restrict__ g,
                                                  float *__restrict__ loss, AdamArgs a)
{
    __shared__ float run[8][32];
    const int lane = threadIdx.x & 31, r = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
    const int per = (blocks + 7) / 8, q0 = r * per, q1 = min(q0 + per, blocks);
    float acc = 0.0f;
    if (i < kPart) {
#pragma unroll 8
        for (int q = q0; q < q1; ++q) acc += part[(int64_t)q * kPart + i];
    }
    run[r][lane] = acc;
    __syncthreads();
    if (r != 0 || i >= kPart) return;
    float gi = 0.0f;
    for (int k = 0; k < 8; ++k) gi += run[k][lane];
    if (i == kParams) {
        *loss = gi;
        return;
    }
    g[i] = gi;
    if (!a.w) return;
    const float mi = a.b1 * a.m[i] + (1.0f - a.b1) * gi;
    const float vi = a.b2 * a.v[i] + (1.0f - a.b2) * gi * gi;
    a.m[i] = mi;
    a.v[i] = vi;
    const float wi = a.w[i] - a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + a.eps);
    a.w[i] = wi;
    a.wb[i] = __float2bfloat16_rn(wi);
}

__global__ void to_bf16_kernel(const float *__restrict__ w, __nv_bfloat16 *__restrict__ wb, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) wb[i] = __float2bfloat16_rn(w[i]);
}

int blocks_for(int64_t n, int t)
{
    int64_t b = (n + t - 1) / t;
    return (int)(b < 1 ? 1 : (b > 152 * 8 ? 152 * 8 : b));
}

}  // namespace

struct mm_mlp {
    float *w = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;  // FP32 master, gradient, Adam moments
    __nv_bfloat16 *wb = nullptr;                                  // BF16 compute copy
    float *mu = nullptr, *sd = nullptr;                           // feature standardisation (device)
    float y_mu = 0.0f, y_sd = 1.0f;                               // target standardisation
    int64_t steps = 0;                                            // Adam steps taken
    // work buffers: samples and targets (or predictions) for cap samples, the
    // blocks' gradient sums, the losses of epochs
    int64_t cap = 0;
    float *x = nullptr, *y = nullptr, *part = nullptr, *loss = nullptr;
    int64_t loss_cap = 0;
};

namespace {

void free_work(mm_mlp *p)
{
    for (float *q : {p->x, p->y, p->part, p->loss}) cudaFree(q);
    p->x = p->y = p->part = p->loss = nullptr;
    p->cap = p->loss_cap = 0;
}

mm_status ensure_work(mm_mlp *p, int64_t n, int64_t losses)
{
    if (n <= p->cap && losses <= p->loss_cap) return MM_OK;
    n = n > p->cap ? n : p->cap;
    losses = losses > p->loss_cap ? losses : p->loss_cap;
    free_work(p);
    const size_t f = sizeof(float);
    if (cudaMalloc(&p->x, (size_t)n * kIn * f) != cudaSuccess || cudaMalloc(&p->y, (size_t)n * f) != cudaSuccess ||
        cudaMalloc(&p->part, (size_t)kMaxPart * kPart * f) != cudaSuccess ||
        cudaMalloc(&p->loss, (size_t)losses * f) != cudaSuccess) {
        cudaGetLastError();
        free_work(p);
        return MM_ENOMEM;
    }
    p->cap = n;
    p->loss_cap = losses;
    return MM_OK;
}

Model model_of(const mm_mlp *p) { return {p->wb, p->mu, p->sd, p->y_mu, p->y_sd}; }

// gradient (into p->g) and loss of the n samples in p->x, p->y, and one Adam
// step where a.w is set
mm_status loss_grad(mm_mlp *p, int64_t n, float *loss, const AdamArgs &a)
{
    if (cudaFuncSetAttribute(loss_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GradSmem)) !=
        cudaSuccess)
        return MM_ECUDA;
    const int64_t tiles = (n + kTile - 1) / kTile;
    const int blocks = (int)(tiles < kMaxPart ? tiles : kMaxPart);
    loss_grad_kernel<<<blocks, kGradThreads, sizeof(GradSmem)>>>(model_of(p), p->x, p->y, n, p->part);
    sum_kernel<<<(kPart + 31) / 32, 256>>>(p->part, blocks, p->g, loss, a);
    return cudaGetLastError() == cudaSuccess ? MM_OK : MM_ECUDA;
}

mm_status upload(mm_mlp *p, const float *X, const float *y, int64_t n)
{
    if (cudaMemcpy(p->x, X, (size_t)n * kIn * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess) return MM_ECUDA;
    if (y && cudaMemcpy(p->y, y, (size_t)n * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess) return MM_ECUDA;
    return MM_OK;
}

}  // namespace

extern "C" {

mm_status mm_mlp_create(uint64_t seed, mm_mlp **out)
{
    if (!out) return MM_EINVAL;
    *out = nullptr;
    mm_mlp *p = new (std::nothrow) mm_mlp();
    if (!p) return MM_ENOMEM;
    const size_t f = sizeof(float);
    if (cudaMalloc(&p->w, kParams * f) != cudaSuccess || cudaMalloc(&p->g, kParams * f) != cudaSuccess ||
        cudaMalloc(&p->m, kParams * f) != cudaSuccess || cudaMalloc(&p->v, kParams * f) != cudaSuccess ||
        cudaMalloc(&p->wb, kParams * sizeof(__nv_bfloat16)) != cudaSuccess || cudaMalloc(&p->mu, kIn * f) != cudaSuccess ||
        cudaMalloc(&p->sd, kIn * f) != cudaSuccess) {
        cudaGetLastError();
        mm_mlp_destroy(p);
        return MM_ENOMEM;
    }
    // He-uniform initial weights, zero biases (host generator, seeded)
    std::vector<float> w(kParams, 0.0f);
    std::mt19937_64 rng(seed);
    auto fill = [&](int off, int rows, int cols) {
        const float a = std::sqrt(6.0f / (float)cols);
        std::uniform_real_distribution<float> U(-a, a);
        for (int i = 0; i < rows * cols; ++i) w[(size_t)(off + i)] = U(rng);
    };
    fill(kOffW1, kH, kIn);
    fill(kOffW2, kH, kH);
    fill(kOffW3, 1, kH);
    std::vector<float> ones(kIn, 1.0f), zeros(kIn, 0.0f);
    mm_status st = mm_mlp_set_params(p, w.data(), kParams);
    if (st == MM_OK && (cudaMemcpy(p->mu, zeros.data(), kIn * f, cudaMemcpyHostToDevice) != cudaSuccess ||
                        cudaMemcpy(p->sd, ones.data(), kIn * f, cudaMemcpyHostToDevice) != cudaSuccess))
        st = MM_ECUDA;
    if (st != MM_OK) {
        mm_mlp_destroy(p);
        return st;
    }
    *out = p;
    return MM_OK;
}

mm_status mm_mlp_set_params(mm_mlp *p, const float *params, int64_t n)
{
    if (!p || !params || n != kParams) return MM_EINVAL;
    if (cudaMemcpy(p->w, params, kParams * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess) return MM_ECUDA;
    if (cudaMemset(p->m, 0, kParams * sizeof(float)) != cudaSuccess ||
        cudaMemset(p->v, 0, kParams * sizeof(float)) != cudaSuccess)
        return MM_ECUDA;
    to_bf16_kernel<<<blocks_for(kParams, 256), 256>>>(p->w, p->wb, kParams);
    p->steps = 0;
    return cudaDeviceSynchronize() == cudaSuccess ? MM_OK : MM_ECUDA;
}

mm_status mm_mlp_get_params(mm_mlp *p, float *params, int64_t n)
{
    if (!p || !params || n < kParams) return MM_EINVAL;
    return cudaMemcpy(params, p->w, kParams * sizeof(float), cudaMemcpyDeviceToHost) == cudaSuccess ? MM_OK : MM_ECUDA;
}

mm_status mm_mlp_set_normalisation(mm_mlp *p, const float *mu, const float *sd, float y_mu, float y_sd)
{
    if (!p || !mu || !sd || !(y_sd > 0.0f)) return MM_EINVAL;
    for (int k = 0; k < kIn; ++k)
        if (!(sd[k] > 0.0f)) return MM_EINVAL;
    if (cudaMemcpy(p->mu, mu, kIn * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(p->sd, sd, kIn * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess)
        return MM_ECUDA;
    p->y_mu = y_mu;
    p->y_sd = y_sd;
    return MM_OK;
}

mm_status mm_mlp_loss_grad(mm_mlp *p, const float *X, const float *y, int64_t n, float *loss, float *grad,
                           int64_t grad_cap)
{
    if (!p || !X || !y || n < 1 || !loss || (grad && grad_cap < kParams)) return MM_EINVAL;
    mm_status st = ensure_work(p, n, 1);
    if (st != MM_OK) return st;
    if ((st = upload(p, X, y, n)) != MM_OK) return st;
    if ((st = loss_grad(p, n, p->loss, AdamArgs{})) != MM_OK) return st;
    if (cudaMemcpy(loss, p->loss, sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess) return MM_ECUDA;
    if (grad && cudaMemcpy(grad, p->g, kParams * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess) return MM_ECUDA;
    return cudaGetLastError() == cudaSuccess ? MM_OK : MM_ECUDA;
}

mm_status mm_mlp_train(mm_mlp *p, const float *X, const float *y, int64_t n, int32_t epochs, float lr,
                       float *loss_per_epoch)
{
    if (!p || !X || !y || n < 2 || epochs < 0 || !(lr > 0.0f)) return MM_EINVAL;
    // standardisation from the training set
    float mu[kIn], sd[kIn];
    for (int k = 0; k < kIn; ++k) {
        double s1 = 0.0, s2 = 0.0;
        for (int64_t s = 0; s < n; ++s) {
            const double v = X[s * kIn + k];
            s1 += v;
            s2 += v * v;
        }
        const double m = s1 / (double)n, var = s2 / (double)n - m * m;
        mu[k] = (float)m;
        sd[k] = (float)(var > 1e-12 ? std::sqrt(var) : 1.0);
    }
    double t1 = 0.0, t2 = 0.0;
    for (int64_t s = 0; s < n; ++s) {
        t1 += y[s];
        t2 += (double)y[s] * y[s];
    }
    const double ym = t1 / (double)n, yv = t2 / (double)n - ym * ym;
    mm_status st = mm_mlp_set_normalisation(p, mu, sd, (float)ym, (float)(yv > 1e-24 ? std::sqrt(yv) : 1.0));
    if (st != MM_OK) return st;
    if ((st = ensure_work(p, n, epochs > 0 ? epochs : 1)) != MM_OK) return st;
    if ((st = upload(p, X, y, n)) != MM_OK) return st;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    for (int32_t e = 0; e < epochs; ++e) {
        p->steps++;
        const float c1 = 1.0f - std::pow(b1, (float)p->steps), c2 = 1.0f - std::pow(b2, (float)p->steps);
        if ((st = loss_grad(p, n, p->loss + e, AdamArgs{p->w, p->m, p->v, p->wb, lr, b1, b2, eps, c1, c2})) != MM_OK) return st;
    }
    if (loss_per_epoch && epochs > 0 &&
        cudaMemcpy(loss_per_epoch, p->loss, (size_t)epochs * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess)
        return MM_ECUDA;
    return cudaDeviceSynchronize() == cudaSuccess && cudaGetLastError() == cudaSuccess ? MM_OK : MM_ECUDA;
}

mm_status mm_mlp_predict(mm_mlp *p, const float *X, int64_t n, float *out)
{
    if (!p || !X || !out || n < 1) return MM_EINVAL;
    mm_status st = ensure_work(p, n, 1);
    if (st != MM_OK) return st;
    if ((st = upload(p, X, nullptr, n)) != MM_OK) return st;
    predict_kernel<<<blocks_for(n, kFwdThreads * kFwdSamples), kFwdThreads>>>(model_of(p), p->x, n, p->y);
    if (cudaGetLastError() != cudaSuccess) return MM_ECUDA;
    if (cudaMemcpy(out, p->y, (size_t)n * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess) return MM_ECUDA;
    return MM_OK;
}

void mm_mlp_destroy(mm_mlp *p)
{
    if (!p) return;
    free_work(p);
    for (void *q : {(void *)p->w, (void *)p->g, (void *)p->m, (void *)p->v, (void *)p->wb, (void *)p->mu, (void *)p->sd})
        cudaFree(q);
    delete p;
}

}  // extern "C"
