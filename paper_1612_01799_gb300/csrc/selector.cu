// Learned grid selection: features of a coarse density sample and a small MLP that maps
// them to the predicted log10 error of the solver at each candidate grid size.
//
// Features (one block per density): the 32^3 sample's discrete Fourier transform, its
// power |F|^2 averaged over 64 radial shells of |k| in [0, 16 sqrt 3], as
// log10(P_b / P_0) clamped to [-30, 0].  The transform is three passes of 32-point DFTs
// over shared memory (x: real input, 17 bins kept; y and z: complex).
//
// MLP: 64 -> 64 -> 64 -> 64 -> K with ReLU on the hidden layers, FP32.  Parameters in one
// array: W1 (64x64), b1, W2 (64x64), b2, W3 (64x64), b3, W4 (K x 64), b4; W[j][i] multiplies
// input i into unit j.  Training kernels: forward (keeping the hidden activations), loss
// gradient of the mean squared error, backward (parameter gradients summed per block, the
// blocks added with atomics), Adam.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "../../include/poisson.h"
#include "solver.h"

namespace {

constexpr int kS = 32;        // sample points per axis
constexpr int kX = kS / 2 + 1;  // kept x bins of the real transform
constexpr int kBins = POISSON_FEATURES;
constexpr int kH = 64;        // hidden width
constexpr int kMaxK = POISSON_MAX_CANDIDATES;

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

__global__ void __launch_bounds__(512) k_features(const float *__restrict__ sample, float *__restrict__ feat) {
    extern __shared__ float2 F[];  // [z][y][kx], kX bins of x
    __shared__ float2 W[kS];       // exp(-2 pi i m / 32)
    __shared__ float pw[kBins], cnt[kBins];
    const float *x = sample + (size_t)blockIdx.x * kS * kS * kS;
    for (int m = threadIdx.x; m < kS; m += blockDim.x) {
        double sn, cs;
        sincospi(-2.0 * m / kS, &sn, &cs);
        W[m] = make_float2((float)cs, (float)sn);
    }
    for (int b = threadIdx.x; b < kBins; b += blockDim.x) pw[b] = cnt[b] = 0.f;
    __syncthreads();
    // x: each (y, z) row, real input -> bins 0..16.
    for (int i = threadIdx.x; i < kS * kS * kX; i += blockDim.x) {
        const int k = i % kX, row = i / kX;
        const float *r = x + (size_t)row * kS;
        float2 acc = make_float2(0.f, 0.f);
        for (int n = 0; n < kS; ++n) {
            const float2 w = W[(n * k) % kS];
            acc.x += r[n] * w.x;
            acc.y += r[n] * w.y;
        }
        F[i] = acc;
    }
    __syncthreads();
    // y: columns (z, kx) over y, in place through registers of the column.
    for (int c = threadIdx.x; c < kS * kX; c += blockDim.x) {
        const int z = c / kX, kx = c % kX;
        float2 col[kS];
        for (int y = 0; y < kS; ++y) col[y] = F[(z * kS + y) * kX + kx];
        for (int ky = 0; ky < kS; ++ky) {
            float2 acc = make_float2(0.f, 0.f);
            for (int y = 0; y < kS; ++y) {
                const float2 t = cmul(col[y], W[(y * ky) % kS]);
                acc.x += t.x;
                acc.y += t.y;
            }
            F[(z * kS + ky) * kX + kx] = acc;
        }
    }
    __syncthreads();
    // z: columns (ky, kx) over z; power into radial shells.
    const float kmax = 16.f * 1.7320508075688772f;
    for (int c = threadIdx.x; c < kS * kX; c += blockDim.x) {
        const int ky = c / kX, kx = c % kX;
        float2 col[kS];
        for (int z = 0; z < kS; ++z) col[z] = F[(z * kS + ky) * kX + kx];
        const int sky = ky < kS / 2 ? ky : ky - kS;
        const float wgt = (kx == 0 || kx == kS / 2) ? 1.f : 2.f;
        for (int kz = 0; kz < kS; ++kz) {
            float2 acc = make_float2(0.f, 0.f);
            for (int z = 0; z < kS; ++z) {
                const float2 t = cmul(col[z], W[(z * kz) % kS]);
                acc.x += t.x;
                acc.y += t.y;
            }
            const int skz = kz < kS / 2 ? kz : kz - kS;
            const float kr = sqrtf((float)(kx * kx + sky * sky + skz * skz));
            int b = (int)(kr / kmax * kBins);
            b = b < kBins ? b : kBins - 1;
            atomicAdd(&pw[b], wgt * (acc.x * acc.x + acc.y * acc.y));
            atomicAdd(&cnt[b], wgt);
        }
    }
    __syncthreads();
    for (int b = threadIdx.x; b < kBins; b += blockDim.x) {
        const float p0 = pw[0] / fmaxf(cnt[0], 1.f);
        const float pb = cnt[b] > 0.f ? pw[b] / cnt[b] : 0.f;
        float v = log10f(pb / fmaxf(p0, 1e-37f) + 1e-30f);
        feat[(size_t)blockIdx.x * kBins + b] = fminf(fmaxf(v, -30.f), 0.f);
    }
}

// Offsets of the parameter blocks for K outputs.
__host__ __device__ inline int off_w(int l) { return l * (kH * kH + kH); }
__host__ __device__ inline int off_b(int l) { return l * (kH * kH + kH) + kH * kH; }
__host__ __device__ inline int nparams(int K) { return 3 * (kH * kH + kH) + K * kH + K; }

// Samples per block of the forward and backward passes: a block stages the weights in shared
// memory once for all its samples, thread (j, sample) makes unit j.
constexpr int kFwdT = 4, kBwdT = 8, kNT = 256;
constexpr int kWP = kH + 1;  // pitch of a transposed weight matrix

// acts: B x 3 x 64 hidden activations (may be null).  The weights of all layers come in with
// coalesced loads, transposed so that the units of a warp read neighbouring words (one block
// per sample with each thread walking its own row of W took 23 us for 384 samples; 10.5 us here).
__global__ void __launch_bounds__(kNT) k_forward(const float *__restrict__ p, int K, const float *__restrict__ x,
                                                 int count, float *__restrict__ y, float *__restrict__ acts) {
    extern __shared__ float sw[];  // W1^T, W2^T, W3^T, W4^T
    __shared__ float h[2][kFwdT][kH];
    const int j = threadIdx.x % kH, t = threadIdx.x / kH, b = blockIdx.x * kFwdT + t;
    for (int l = 0; l < 3; ++l)
#pragma unroll
        for (int e = threadIdx.x; e < kH * kH; e += kNT) sw[l * kH * kWP + (e % kH) * kWP + e / kH] = p[off_w(l) + e];
    for (int e = threadIdx.x; e < K * kH; e += kNT) sw[3 * kH * kWP + (e % kH) * kWP + e / kH] = p[off_w(3) + e];
    h[0][t][j] = b < count ? x[(size_t)b * kH + j] : 0.f;
    __syncthreads();
    int cur = 0;
    for (int l = 0; l < 3; ++l) {
        const float *W = sw + l * kH * kWP + j;
        float a = p[off_b(l) + j];
#pragma unroll 16
        for (int i = 0; i < kH; ++i) a += W[i * kWP] * h[cur][t][i];
        a = fmaxf(a, 0.f);
        if (acts && b < count) acts[((size_t)b * 3 + l) * kH + j] = a;
        h[1 - cur][t][j] = a;
        __syncthreads();
        cur = 1 - cur;
    }
    if (j < K && b < count) {
        const float *W = sw + 3 * kH * kWP + j;
        float a = p[off_w(3) + K * kH + j];
#pragma unroll 16
        for (int i = 0; i < kH; ++i) a += W[i * kWP] * h[cur][t][i];
        y[(size_t)b * K + j] = a;
    }
}
constexpr int kFwdSmem = 4 * kH * kWP * (int)sizeof(float);

// dy = 2 (y - t) / (B K) and the loss sum (y - t)^2 / (B K) (one block).
constexpr int kLossNT = 1024;
__global__ void __launch_bounds__(kLossNT) k_loss(const float *__restrict__ y, const float *__restrict__ t, int n,
                                                  float *__restrict__ dy, float *__restrict__ loss) {
    __shared__ float s[kLossNT / 32];
    float acc = 0.f;
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += kLossNT) {
        const float d = y[i] - t[i];
        dy[i] = 2.f * d / n;
        acc += d * d;
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (threadIdx.x % 32 == 0) s[threadIdx.x / 32] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        acc = s[threadIdx.x];
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (threadIdx.x == 0) *loss = acc / n;
    }
}

// g[0..3] += v, in one reduction where g is 16-byte aligned.
__device__ __forceinline__ void add4(float *g, float4 v, bool vec) {
    if (vec) {
        atomicAdd(reinterpret_cast<float4 *>(g), v);
    } else {
        atomicAdd(g, v.x);
        atomicAdd(g + 1, v.y);
        atomicAdd(g + 2, v.z);
        atomicAdd(g + 3, v.w);
    }
}

// A block takes kBwdT samples: their deltas back through the layers, then its part of each
// weight gradient, sum_b delta_j a_i, as a 4 x 4 tile per thread summed in registers over the
// samples, added to g with one 16-byte reduction per row (vec: g is 16-byte aligned).  One
// atomic per sample and parameter, as before, is 5 million at 13 thousand addresses for 384
// samples: 97 us, 12 us here.
__global__ void __launch_bounds__(kNT) k_backward(const float *__restrict__ p, int K, const float *__restrict__ x,
                                                  const float *__restrict__ acts, int count,
                                                  const float *__restrict__ dy, float *__restrict__ g, bool vec) {
    __shared__ __align__(16) float a[4][kBwdT][kH];  // layer inputs: x, h1, h2, h3
    __shared__ __align__(16) float d[3][kBwdT][kH];  // deltas of layers 1, 2, 3
    __shared__ float e[kBwdT][kMaxK];
    __shared__ float W[2][kH * kH];                  // W2, W3
    const int tid = threadIdx.x, j = tid % kH, b0 = blockIdx.x * kBwdT, nb = min(kBwdT, count - b0);
#pragma unroll
    for (int l = 1; l < 3; ++l)
        for (int i = tid; i < kH * kH; i += kNT) W[l - 1][i] = p[off_w(l) + i];
    for (int t = tid / kH; t < kBwdT; t += kNT / kH) {
        const bool ok = t < nb;
        a[0][t][j] = ok ? x[(size_t)(b0 + t) * kH + j] : 0.f;
        for (int l = 0; l < 3; ++l) a[l + 1][t][j] = ok ? acts[((size_t)(b0 + t) * 3 + l) * kH + j] : 0.f;
        if (j < K) e[t][j] = ok ? dy[(size_t)(b0 + t) * K + j] : 0.f;
    }
    __syncthreads();
    for (int t = tid / kH; t < kBwdT; t += kNT / kH) {
        float acc = 0.f;
        for (int k = 0; k < K; ++k) acc += p[off_w(3) + k * kH + j] * e[t][k];
        d[2][t][j] = a[3][t][j] > 0.f ? acc : 0.f;
    }
    __syncthreads();
    for (int l = 2; l > 0; --l) {
        for (int t = tid / kH; t < kBwdT; t += kNT / kH) {
            float s = 0.f;
#pragma unroll 16
            for (int k = 0; k < kH; ++k) s += W[l - 1][k * kH + j] * d[l][t][k];
            d[l - 1][t][j] = a[l][t][j] > 0.f ? s : 0.f;
        }
        __syncthreads();
    }
    const int r0 = 4 * (tid / 16), c0 = 4 * (tid % 16);
    for (int l = 0; l < 3; ++l) {
        float4 acc[4] = {};
#pragma unroll
        for (int t = 0; t < kBwdT; ++t) {
            const float4 av = *reinterpret_cast<const float4 *>(&a[l][t][c0]);
            const float4 dv = *reinterpret_cast<const float4 *>(&d[l][t][r0]);
            const float dr[4] = {dv.x, dv.y, dv.z, dv.w};
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                acc[r].x += dr[r] * av.x;
                acc[r].y += dr[r] * av.y;
                acc[r].z += dr[r] * av.z;
                acc[r].w += dr[r] * av.w;
            }
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) add4(g + off_w(l) + (r0 + r) * kH + c0, acc[r], vec);
    }
    if (tid / 16 < K) {  // output layer: row tid / 16
        const int k = tid / 16;
        float4 acc = {};
#pragma unroll
        for (int t = 0; t < kBwdT; ++t) {
            const float4 av = *reinterpret_cast<const float4 *>(&a[3][t][c0]);
            acc.x += e[t][k] * av.x;
            acc.y += e[t][k] * av.y;
            acc.z += e[t][k] * av.z;
            acc.w += e[t][k] * av.w;
        }
        add4(g + off_w(3) + k * kH + c0, acc, vec);
    }
    for (int i = tid; i < 3 * kH + K; i += kNT) {  // biases
        float s = 0.f;
#pragma unroll
        for (int t = 0; t < kBwdT; ++t) s += i < 3 * kH ? d[i / kH][t][i % kH] : e[t][i - 3 * kH];
        atomicAdd(i < 3 * kH ? g + off_b(i / kH) + i % kH : g + off_w(3) + K * kH + i - 3 * kH, s);
    }
}

__global__ void k_adam(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m, float *__restrict__ v,
                       int n, float lr, float b1, float b2, float eps, float c1, float c2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi, vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

int ok(cudaError_t e) {
    gsp::note_cuda_error(e);
    return e == cudaSuccess ? POISSON_OK : POISSON_ERR_CUDA;
}

}  // namespace

extern "C" int poisson_features32(const float *sample_d, int count, float *feat_d, void *stream) {
    if (count < 0 || (count > 0 && (!sample_d || !feat_d))) return POISSON_ERR_ARG;
    if (count == 0) return POISSON_OK;
    const size_t smem = (size_t)kS * kS * kX * sizeof(float2);
    cudaError_t e = cudaFuncSetAttribute(k_features, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return ok(e);
    k_features<<<count, 512, smem, (cudaStream_t)stream>>>(sample_d, feat_d);
    return ok(cudaGetLastError());
}

extern "C" int poisson_mlp_nparams(int K) { return K >= 1 && K <= kMaxK ? nparams(K) : -1; }

extern "C" int poisson_mlp_forward(const float *params_d, int K, const float *x_d, int count, float *y_d,
                                   float *acts_d, void *stream) {
    if (K < 1 || K > kMaxK || count < 0 || (count > 0 && (!params_d || !x_d || !y_d))) return POISSON_ERR_ARG;
    if (count == 0) return POISSON_OK;
    const cudaError_t e = cudaFuncSetAttribute(k_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, kFwdSmem);
    if (e != cudaSuccess) return ok(e);
    k_forward<<<(count + kFwdT - 1) / kFwdT, kNT, kFwdSmem, (cudaStream_t)stream>>>(params_d, K, x_d, count, y_d, acts_d);
    return ok(cudaGetLastError());
}

extern "C" int poisson_mlp_loss(const float *y_d, const float *target_d, int n, float *dy_d, float *loss_d,
                                void *stream) {
    if (n < 1 || !y_d || !target_d || !dy_d || !loss_d) return POISSON_ERR_ARG;
    k_loss<<<1, kLossNT, 0, (cudaStream_t)stream>>>(y_d, target_d, n, dy_d, loss_d);
    return ok(cudaGetLastError());
}

extern "C" int poisson_mlp_backward(const float *params_d, int K, const float *x_d, const float *acts_d,
                                    int count, const float *dy_d, float *grad_d, void *stream) {
    if (K < 1 || K > kMaxK || count < 0 || (count > 0 && (!params_d || !x_d || !acts_d || !dy_d || !grad_d)))
        return POISSON_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e = cudaMemsetAsync(grad_d, 0, sizeof(float) * nparams(K), s);
    if (e != cudaSuccess || count == 0) return ok(e);
    const bool vec = reinterpret_cast<uintptr_t>(grad_d) % 16 == 0;
    k_backward<<<(count + kBwdT - 1) / kBwdT, kNT, 0, s>>>(params_d, K, x_d, acts_d, count, dy_d, grad_d, vec);
    return ok(cudaGetLastError());
}

extern "C" int poisson_mlp_adam(float *params_d, const float *grad_d, float *m_d, float *v_d, int n, float lr,
                                float beta1, float beta2, float eps, int step, void *stream) {
    if (n < 1 || step < 1 || !params_d || !grad_d || !m_d || !v_d) return POISSON_ERR_ARG;
    const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
    k_adam<<<(n + 255) / 256, 256, 0, (cudaStream_t)stream>>>(params_d, grad_d, m_d, v_d, n, lr, beta1, beta2,
                                                               eps, c1, c2);
    return ok(cudaGetLastError());
}

// ---- selector objects -------------------------------------------------------------------
// File (little endian): "GSPSEL01", int32 K, int32 N[K], float margin, float feat_mean[64],
// float feat_std[64], float params[nparams(K)].  The network predicts log10 of the relative
// L2 error of a solve at each candidate N from the standardised features.

#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

struct poisson_selector_s {
    int K = 0;
    int N[kMaxK] = {};
    float margin = 0.f;
    int capacity = 0;
    float *params = nullptr, *mean = nullptr, *stdv = nullptr;  // device
    float *feat = nullptr, *pred = nullptr;                      // device, capacity rows
};

namespace {
__global__ void k_standardise(float *__restrict__ f, const float *__restrict__ mean, const float *__restrict__ sd,
                              int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) f[i] = (f[i] - mean[i % kBins]) / sd[i % kBins];
}
void free_selector(poisson_selector s) {
    if (!s) return;
    float *bufs[] = {s->params, s->mean, s->stdv, s->feat, s->pred};
    for (float *b : bufs)
        if (b) cudaFree(b);
    delete s;
}
}  // namespace

extern "C" int poisson_selector_load(poisson_selector *out, const char *path, int capacity) {
    if (!out || !path || capacity < 1) return POISSON_ERR_ARG;
    *out = nullptr;
    FILE *f = std::fopen(path, "rb");
    if (!f) return POISSON_ERR_ARG;
    char magic[8];
    poisson_selector s = new (std::nothrow) poisson_selector_s();
    if (!s) {
        std::fclose(f);
        return POISSON_ERR_ALLOC;
    }
    bool good = std::fread(magic, 1, 8, f) == 8 && std::memcmp(magic, "GSPSEL01", 8) == 0 &&
                std::fread(&s->K, 4, 1, f) == 1 && s->K >= 1 && s->K <= kMaxK &&
                std::fread(s->N, 4, s->K, f) == (size_t)s->K && std::fread(&s->margin, 4, 1, f) == 1;
    std::vector<float> mean(kBins), sd(kBins), params;
    if (good) {
        params.resize(nparams(s->K));
        good = std::fread(mean.data(), 4, kBins, f) == (size_t)kBins &&
               std::fread(sd.data(), 4, kBins, f) == (size_t)kBins &&
               std::fread(params.data(), 4, params.size(), f) == params.size();
    }
    std::fclose(f);
    if (!good) {
        delete s;
        return POISSON_ERR_ARG;
    }
    s->capacity = capacity;
    auto alloc = [&](float **p, size_t n) { return cudaMalloc(p, n * sizeof(float)) == cudaSuccess; };
    if (!alloc(&s->params, params.size()) || !alloc(&s->mean, kBins) || !alloc(&s->stdv, kBins) ||
        !alloc(&s->feat, (size_t)capacity * kBins) || !alloc(&s->pred, (size_t)capacity * s->K)) {
        free_selector(s);
        return POISSON_ERR_ALLOC;
    }
    if (cudaMemcpy(s->params, params.data(), params.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(s->mean, mean.data(), kBins * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(s->stdv, sd.data(), kBins * 4, cudaMemcpyHostToDevice) != cudaSuccess) {
        free_selector(s);
        return POISSON_ERR_CUDA;
    }
    *out = s;
    return POISSON_OK;
}

extern "C" int poisson_selector_destroy(poisson_selector s) {
    free_selector(s);
    return POISSON_OK;
}

extern "C" int poisson_select_n(poisson_selector s, const float *sample32_d, int count, double tol, int *N_out,
                                float *pred_out, void *stream) {
    if (!s || !sample32_d || !N_out || count < 1 || count > s->capacity || !(tol > 0.0)) return POISSON_ERR_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    int rc = poisson_features32(sample32_d, count, s->feat, stream);
    if (rc) return rc;
    const int n = count * kBins;
    k_standardise<<<(n + 255) / 256, 256, 0, st>>>(s->feat, s->mean, s->stdv, n);
    if ((rc = poisson_mlp_forward(s->params, s->K, s->feat, count, s->pred, nullptr, stream))) return rc;
    std::vector<float> pred((size_t)count * s->K);
    if (cudaMemcpyAsync(pred.data(), s->pred, pred.size() * 4, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return POISSON_ERR_CUDA;
    const float goal = (float)std::log10(tol) - s->margin;
    for (int b = 0; b < count; ++b) {
        int pick = s->N[s->K - 1];
        for (int k = 0; k < s->K; ++k)
            if (pred[(size_t)b * s->K + k] <= goal) {
                pick = s->N[k];
                break;
            }
        N_out[b] = pick;
    }
    if (pred_out) std::memcpy(pred_out, pred.data(), pred.size() * 4);
    return POISSON_OK;
}
