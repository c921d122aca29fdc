// Learned chemical-potential seed: spectral-moment features of (H, S) and a small MLP with
// hand-written forward, backward and Adam kernels (FP32).  The paper searches mu iteratively
// (Sec. II.C.3); this network only proposes the starting bracket for that search.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <string>
#include <vector>

#include "ndsi.h"
#include "plan.hpp"

namespace ndsi {
namespace {

constexpr int kIn = NDSI_MLP_INPUTS, kHid = NDSI_MLP_HIDDEN;
constexpr int kNW1 = kHid * kIn, kNB1 = kHid, kNW2 = kHid * kHid, kNB2 = kHid, kNW3 = kHid, kNB3 = 1;
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kNW1, kOffW2 = kOffB1 + kNB1, kOffB2 = kOffW2 + kNW2,
              kOffW3 = kOffB2 + kNB2, kOffB3 = kOffW3 + kNW3, kNParams = kOffB3 + kNB3;
static_assert(kNParams == NDSI_MLP_PARAMS, "parameter layout");
constexpr int kBatchBlock = 16;  // samples a CTA of the gradient kernel takes at a time: 125 CTAs for 2000 samples
// CTAs of the gradient kernel at most (four fit an SM): each then takes several groups of samples, so that the
// partial gradients stay within 15 MB for any number of samples.
constexpr int kGradBlocks = 4 * 152;
inline int grad_blocks(int n) { return std::min(n / kBatchBlock + (n % kBatchBlock != 0), kGradBlocks); }

// SplitMix64 (Steele, Lea, Flood 2014) as a counter-based generator.
__host__ __device__ inline uint64_t splitmix64(uint64_t x) {
    x += 0x9E3779B97F4A7C15ull;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
    return x ^ (x >> 31);
}
__device__ inline float uniform01(uint64_t seed, uint64_t i) {
    return static_cast<float>((splitmix64(seed ^ splitmix64(i)) >> 40) * (1.0 / 16777216.0));
}

// ------------------------------------------------------------------------ features -----------
// y(:, r) = c1 * (A x(:, r)) + c0 * x(:, r) - cp * p(:, r) for R vectors stored row-major
// [n][R]; A = (vals - shift*I) / scale on the CSR pattern.  Also partial sums of z . y per block
// (z = the Rademacher start vectors) for the stochastic trace.
__global__ void __launch_bounds__(256) k_cheb_step(const int64_t* __restrict__ rowptr,
                                                   const int32_t* __restrict__ col,
                                                   const double* __restrict__ vals, double shift,
                                                   double scale, int64_t n, int R,
                                                   const float* __restrict__ x,
                                                   const float* __restrict__ prev, float c1, float cp,
                                                   float* __restrict__ y, uint64_t seed,
                                                   double* __restrict__ partial) {
    __shared__ double red[256];
    const int64_t idx = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
    double dot = 0.0;
    if (idx < n * R) {
        const int64_t i = idx / R;
        const int r = static_cast<int>(idx % R);
        float acc = 0.f;
        for (int64_t k = rowptr[i]; k < rowptr[i + 1]; ++k) {
            const int64_t j = col[k];
            float a = static_cast<float>(vals[k]);
            if (j == i) a -= static_cast<float>(shift);
            acc += a * x[j * R + r];
        }
        acc = acc / static_cast<float>(scale);
        const float v = c1 * acc - (prev ? cp * prev[idx] : 0.f);
        y[idx] = v;
        const float z = (splitmix64(seed ^ splitmix64(static_cast<uint64_t>(idx))) & 1) ? 1.f : -1.f;
        dot = static_cast<double>(z) * v;
    }
    red[threadIdx.x] = dot;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}

__global__ void k_rademacher(int64_t count, uint64_t seed, float* __restrict__ z) {
    for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < count;
         i += static_cast<int64_t>(gridDim.x) * blockDim.x)
        z[i] = (splitmix64(seed ^ splitmix64(static_cast<uint64_t>(i))) & 1) ? 1.f : -1.f;
}

__global__ void k_sum_partials(const double* __restrict__ partial, int nblocks, double norm,
                               float* __restrict__ out) {
    __shared__ double red[256];
    double v = 0.0;
    for (int i = threadIdx.x; i < nblocks; i += blockDim.x) v += partial[i];
    red[threadIdx.x] = v;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = static_cast<float>(red[0] * norm);
}

// ----------------------------------------------------------------------------- MLP -----------
__device__ __forceinline__ void mlp_forward_one(const float* __restrict__ P, const float* x, float* h1,
                                                float* h2, float& y) {
    for (int j = 0; j < kHid; ++j) {
        float a = P[kOffB1 + j];
        for (int i = 0; i < kIn; ++i) a = fmaf(P[kOffW1 + j * kIn + i], x[i], a);
        h1[j] = tanhf(a);
    }
    for (int j = 0; j < kHid; ++j) {
        float a = P[kOffB2 + j];
        for (int i = 0; i < kHid; ++i) a = fmaf(P[kOffW2 + j * kHid + i], h1[i], a);
        h2[j] = tanhf(a);
    }
    float a = P[kOffB3];
    for (int i = 0; i < kHid; ++i) a = fmaf(P[kOffW3 + i], h2[i], a);
    y = a;
}

__global__ void __launch_bounds__(128) k_mlp_forward(const float* __restrict__ params,
                                                     const float* __restrict__ X, int n,
                                                     float* __restrict__ Y) {
    __shared__ float P[kNParams];
    for (int i = threadIdx.x; i < kNParams; i += blockDim.x) P[i] = params[i];
    __syncthreads();
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    float x[kIn], h1[kHid], h2[kHid], y;
    for (int i = 0; i < kIn; ++i) x[i] = X[static_cast<int64_t>(s) * kIn + i];
    mlp_forward_one(P, x, h1, h2, y);
    Y[s] = y;
}

// Mean-squared-error gradient of groups of up to 16 samples, summed over a block's groups, one partial gradient per block
// (summed in a fixed order by k_mlp_reduce, so the result is deterministic).  The work is small
// (37 kflop per sample) and latency decides: all 256 threads share every layer (an output neuron and
// four samples each), activations lie neuron-major with the samples as float4, weights row-padded
// against bank conflicts.  A call of 25 training steps on 2000 samples, with k_mlp_reduce: 3.46 -> 0.69 ms (one
// thread per sample over 64-sample blocks left 120 SMs idle and ran 37 kflop serially).
struct MlpShared {
    float w1[kHid][kIn + 1], w2[kHid][kHid + 1], w3[kHid], b1[kHid], b2[kHid], b3;
    float4 x[kIn][kBatchBlock / 4], h1[kHid][kBatchBlock / 4 + 1], h2[kHid][kBatchBlock / 4 + 1];
    float4 dz1[kHid][kBatchBlock / 4 + 1], dz2[kHid][kBatchBlock / 4 + 1];
    float dy[kBatchBlock], l[kBatchBlock];
};
__device__ __forceinline__ void fma4(float4& a, float w, const float4& v) {
    a.x = fmaf(w, v.x, a.x);
    a.y = fmaf(w, v.y, a.y);
    a.z = fmaf(w, v.z, a.z);
    a.w = fmaf(w, v.w, a.w);
}
__device__ __forceinline__ float dot4(const float4& a, const float4& b, float acc) {
    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, acc))));
}
__device__ __forceinline__ float4 tanh4(const float4& v) { return make_float4(tanhf(v.x), tanhf(v.y), tanhf(v.z), tanhf(v.w)); }
// a (1 - h^2) per component
__device__ __forceinline__ float4 dtanh4(const float4& a, const float4& h) {
    return make_float4(a.x * (1.f - h.x * h.x), a.y * (1.f - h.y * h.y), a.z * (1.f - h.z * h.z), a.w * (1.f - h.w * h.w));
}

// ONE: a single group per block (a loop that may come again costs 7% of a call of 25 steps).
template <bool ONE>
__global__ void __launch_bounds__(256) k_mlp_grad(const float* __restrict__ params, const float* __restrict__ X,
                                                  const float* __restrict__ T, int n, float* __restrict__ partial,
                                                  float* __restrict__ loss_partial) {
    extern __shared__ float4 mlp_smem[];
    MlpShared& m = *reinterpret_cast<MlpShared*>(mlp_smem);
    const int tid = threadIdx.x;
    for (int i = tid; i < kNW1; i += 256) m.w1[i / kIn][i % kIn] = params[kOffW1 + i];
    for (int i = tid; i < kNW2; i += 256) m.w2[i / kHid][i % kHid] = params[kOffW2 + i];
    if (tid < kHid) {
        m.b1[tid] = params[kOffB1 + tid];
        m.b2[tid] = params[kOffB2 + tid];
        m.w3[tid] = params[kOffW3 + tid];
    }
    if (tid == 0) m.b3 = params[kOffB3];
    const int j = tid % kHid, g = tid / kHid;    // a neuron and a group of four samples
    const int r0 = tid / 16, c0 = tid % 16;      // dW2 = dz2^T h1 in 4 x 4 register tiles, dW1 = dz1^T x in 4 x 2
    float dw2[4][4] = {}, dw1[4][2] = {}, db1 = 0.f, db2 = 0.f, dw3 = 0.f, db3 = 0.f, lsum = 0.f;
    const int groups = n / kBatchBlock + (n % kBatchBlock != 0);
    float* out = partial + static_cast<int64_t>(blockIdx.x) * kNParams;
    for (int grp = blockIdx.x;; grp += gridDim.x) {
        const bool last = ONE || groups - grp <= static_cast<int>(gridDim.x);
        const int s0 = grp * kBatchBlock, nb = min(kBatchBlock, n - s0);
        for (int i = tid; i < kBatchBlock * kIn; i += 256) {
            const int b = i / kIn, k = i % kIn;
            reinterpret_cast<float*>(m.x[k])[b] = b < nb ? X[static_cast<int64_t>(s0 + b) * kIn + k] : 0.f;
        }
        __syncthreads();
        {
            float4 a = make_float4(m.b1[j], m.b1[j], m.b1[j], m.b1[j]);
#pragma unroll 8
            for (int i = 0; i < kIn; ++i) fma4(a, m.w1[j][i], m.x[i][g]);
            m.h1[j][g] = tanh4(a);
        }
        __syncthreads();
        {
            float4 a = make_float4(m.b2[j], m.b2[j], m.b2[j], m.b2[j]);
#pragma unroll 8
            for (int i = 0; i < kHid; ++i) fma4(a, m.w2[j][i], m.h1[i][g]);
            m.h2[j][g] = tanh4(a);
        }
        __syncthreads();
        {
            // output and its error: sixteen threads per sample, four neurons each
            const int b = tid / 16, q = tid % 16;
            float a = 0.f;
#pragma unroll
            for (int u = 0; u < kHid / 16; ++u) a = fmaf(m.w3[q + 16 * u], reinterpret_cast<const float*>(m.h2[q + 16 * u])[b], a);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            if (q == 0) {
                const float e = b < nb ? a + m.b3 - T[s0 + b] : 0.f;
                m.dy[b] = 2.f * e / static_cast<float>(n);
                m.l[b] = e * e / static_cast<float>(n);
            }
        }
        __syncthreads();
        {
            const float4 dy = *reinterpret_cast<const float4*>(&m.dy[4 * g]);
            const float w = m.w3[j];
            m.dz2[j][g] = dtanh4(make_float4(dy.x * w, dy.y * w, dy.z * w, dy.w * w), m.h2[j][g]);
        }
        __syncthreads();
        {
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
            for (int i = 0; i < kHid; ++i) fma4(a, m.w2[i][j], m.dz2[i][g]);
            m.dz1[j][g] = dtanh4(a, m.h1[j][g]);
        }
        __syncthreads();
#pragma unroll
        for (int b = 0; b < kBatchBlock / 4; ++b) {
            float4 u[4], v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                u[q] = m.dz2[r0 + 16 * q][b];
                v[q] = m.h1[c0 + 16 * q][b];
            }
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) dw2[p][q] = dot4(u[p], v[q], dw2[p][q]);
        }
        if (last) {
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) out[kOffW2 + (r0 + 16 * p) * kHid + c0 + 16 * q] = dw2[p][q];
        }
#pragma unroll
        for (int b = 0; b < kBatchBlock / 4; ++b) {
            const float4 v[2] = {m.x[c0][b], m.x[c0 + 16][b]};
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const float4 u = m.dz1[r0 + 16 * p][b];
#pragma unroll
                for (int q = 0; q < 2; ++q) dw1[p][q] = dot4(u, v[q], dw1[p][q]);
            }
        }
        if (last) {
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 2; ++q) out[kOffW1 + (r0 + 16 * p) * kIn + c0 + 16 * q] = dw1[p][q];
        }
        if (tid < kHid) {
#pragma unroll
            for (int b = 0; b < kBatchBlock / 4; ++b) {
                const float4 one = make_float4(1.f, 1.f, 1.f, 1.f);
                db1 = dot4(m.dz1[tid][b], one, db1);
                db2 = dot4(m.dz2[tid][b], one, db2);
                dw3 = dot4(*reinterpret_cast<const float4*>(&m.dy[4 * b]), m.h2[tid][b], dw3);
            }
        }
        if (tid == 0) {
            for (int b = 0; b < kBatchBlock; ++b) {
                db3 += m.dy[b];
                lsum += m.l[b];
            }
        }
        if (last) break;
        __syncthreads();  // the next group's samples take the space
    }
    if (tid < kHid) {
        out[kOffB1 + tid] = db1;
        out[kOffB2 + tid] = db2;
        out[kOffW3 + tid] = dw3;
    }
    if (tid == 0) {
        out[kOffB3] = db3;
        loss_partial[blockIdx.x] = lsum;
    }
}

// Adam's state and step (Kingma and Ba 2015, with bias correction c1, c2).
struct AdamStep {
    float *params, *m, *v;
    float lr, b1, b2, eps, c1, c2;
};

// Sum of the blocks' partial gradients (eight threads per parameter, fixed order), with the Adam step of
// the parameter when `adam.params` is set; block 0 sums the loss.
__global__ void __launch_bounds__(256) k_mlp_reduce(const float* __restrict__ partial, int nblocks,
                                                    float* __restrict__ grad,
                                                    const float* __restrict__ loss_partial,
                                                    float* __restrict__ loss, AdamStep adam) {
    __shared__ float red[8][33];
    const int lane = threadIdx.x & 31, part = threadIdx.x >> 5;
    const int p = blockIdx.x * 32 + lane;
    float a = 0.f;
    if (p < kNParams) {
#pragma unroll 8
        for (int b = part; b < nblocks; b += 8) a += partial[static_cast<int64_t>(b) * kNParams + p];
    }
    red[part][lane] = a;
    __syncthreads();
    if (part == 0 && p < kNParams) {
        float g = 0.f;
#pragma unroll
        for (int q = 0; q < 8; ++q) g += red[q][lane];
        if (grad) grad[p] = g;
        if (adam.params) {
            const float mm = adam.b1 * adam.m[p] + (1.f - adam.b1) * g;
            const float vv = adam.b2 * adam.v[p] + (1.f - adam.b2) * g * g;
            adam.m[p] = mm;
            adam.v[p] = vv;
            adam.params[p] -= adam.lr * (mm / adam.c1) / (sqrtf(vv / adam.c2) + adam.eps);
        }
    }
    if (loss && blockIdx.x == 0 && part == 1) {
        float l = 0.f;
        for (int b = lane; b < nblocks; b += 32) l += loss_partial[b];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (lane == 0) *loss = l;
    }
}

// Glorot-uniform weights, zero biases, from the counter-based generator.
__global__ void k_mlp_init(float* __restrict__ params, uint64_t seed) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= kNParams) return;
    float bound = 0.f;
    if (p < kOffB1) bound = sqrtf(6.f / (kIn + kHid));
    else if (p >= kOffW2 && p < kOffB2) bound = sqrtf(6.f / (kHid + kHid));
    else if (p >= kOffW3 && p < kOffB3) bound = sqrtf(6.f / (kHid + 1));
    params[p] = bound * (2.f * uniform01(seed, static_cast<uint64_t>(p)) - 1.f);
}

int mfail(int code, const std::string& m) {
    set_last_error(m);
    return code;
}

#define MLP_CK(call)                                                                        \
    do {                                                                                    \
        cudaError_t e_ = (call);                                                            \
        if (e_ != cudaSuccess) return mfail(NDSI_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
    } while (0)

bool dev_ptr(const void* p) {
    cudaPointerAttributes a{};
    if (!p || cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

size_t grad_smem() { return sizeof(MlpShared); }

int grad_launch(const float* params, const float* X, const float* T, int n, float* partial, float* lossp,
                float* grad, float* loss, const AdamStep& adam, cudaStream_t st) {
    const int nblk = grad_blocks(n);
    const bool one = n <= kGradBlocks * kBatchBlock;
    (one ? k_mlp_grad<true> : k_mlp_grad<false>)<<<nblk, 256, grad_smem(), st>>>(params, X, T, n, partial, lossp);
    MLP_CK(cudaGetLastError());
    k_mlp_reduce<<<(kNParams + 31) / 32, 256, 0, st>>>(partial, nblk, grad, lossp, loss, adam);
    MLP_CK(cudaGetLastError());
    return NDSI_OK;
}

}  // namespace

int mlp_features(const Plan& P, const double* Hd, const double* Sd, const int64_t* rowptr_d,
                 const int32_t* col_d, double n_electrons, double kT, int R, uint64_t seed, float* feat_d,
                 cudaStream_t st) {
    const int64_t n = P.n;
    const int64_t cnt = n * R;
    float *buf = nullptr;
    double* partial = nullptr;
    const int nblk = static_cast<int>((cnt + 255) / 256);
    MLP_CK(cudaMalloc(&buf, sizeof(float) * cnt * 4));
    if (cudaMalloc(&partial, sizeof(double) * nblk) != cudaSuccess) {
        cudaFree(buf);
        return mfail(NDSI_ERR_OOM, "ndsi_mu_features: scratch allocation failed");
    }
    float* z = buf;
    float* t[3] = {buf + cnt, buf + 2 * cnt, buf + 3 * cnt};
    cudaError_t e = cudaSuccess;
    auto moments = [&](const double* vals, double shift, double scale, int kmax, int out0) {
        // t0 = z, t1 = A z, t_{k+1} = 2 A t_k - t_{k-1}; moment_k = z . t_k / (R n)
        const float* cur = z;
        const float* prv = nullptr;
        for (int k = 1; k <= kmax && e == cudaSuccess; ++k) {
            float* nxt = t[(k - 1) % 3];
            k_cheb_step<<<nblk, 256, 0, st>>>(rowptr_d, col_d, vals, shift, scale, n, R, cur, prv,
                                              k == 1 ? 1.f : 2.f, 1.f, nxt, seed, partial);
            k_sum_partials<<<1, 256, 0, st>>>(partial, nblk, 1.0 / static_cast<double>(cnt), feat_d + out0 + k - 1);
            e = cudaGetLastError();
            prv = cur;
            cur = nxt;
        }
    };
    k_rademacher<<<1024, 256, 0, st>>>(cnt, seed, z);
    e = cudaGetLastError();
    // fixed energy window [-4, 4] Ha for H; S - I in [-0.75, 0.75] for the overlap
    moments(Hd, 0.0, 4.0, 24, 0);
    moments(Sd, 1.0, 0.75, 6, 24);
    const float extra[2] = {static_cast<float>(n_electrons / (2.0 * n)), static_cast<float>(10.0 * kT)};
    if (e == cudaSuccess) e = cudaMemcpyAsync(feat_d + 30, extra, sizeof(extra), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(buf);
    cudaFree(partial);
    if (e != cudaSuccess) return mfail(NDSI_ERR_CUDA, std::string("ndsi_mu_features: ") + cudaGetErrorString(e));
    return NDSI_OK;
}

}  // namespace ndsi

using namespace ndsi;

extern "C" {

int ndsi_mlp_init(float* params, uint64_t seed, void* stream) {
    if (!params || !dev_ptr(params)) return mfail(NDSI_ERR_INVALID, "ndsi_mlp_init: params must be device memory");
    k_mlp_init<<<(kNParams + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream)>>>(params, seed);
    MLP_CK(cudaGetLastError());
    return NDSI_OK;
}

int ndsi_mlp_forward(const float* params, const float* X, int32_t n, float* Y, void* stream) {
    if (!params || !X || !Y || n < 1 || !dev_ptr(params) || !dev_ptr(X) || !dev_ptr(Y))
        return mfail(NDSI_ERR_INVALID, "ndsi_mlp_forward: device arrays and n >= 1 required");
    k_mlp_forward<<<(n + 127) / 128, 128, 0, static_cast<cudaStream_t>(stream)>>>(params, X, n, Y);
    MLP_CK(cudaGetLastError());
    return NDSI_OK;
}

int ndsi_mlp_grad(const float* params, const float* X, const float* T, int32_t n, float* grad, float* loss,
                  void* stream) {
    if (!params || !X || !T || !grad || n < 1 || !dev_ptr(params) || !dev_ptr(X) || !dev_ptr(T) ||
        !dev_ptr(grad) || (loss && !dev_ptr(loss)))
        return mfail(NDSI_ERR_INVALID, "ndsi_mlp_grad: device arrays and n >= 1 required");
    static bool attr = false;
    if (!attr) {
        for (auto f : {&k_mlp_grad<true>, &k_mlp_grad<false>})
            MLP_CK(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(grad_smem())));
        attr = true;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int nblk = grad_blocks(n);
    float *partial = nullptr, *lossp = nullptr;
    MLP_CK(cudaMalloc(&partial, sizeof(float) * (static_cast<size_t>(nblk) * kNParams + nblk)));
    lossp = partial + static_cast<size_t>(nblk) * kNParams;
    int rc = grad_launch(params, X, T, n, partial, lossp, grad, loss, AdamStep{}, st);
    cudaError_t e = cudaStreamSynchronize(st);
    cudaFree(partial);
    if (rc) return rc;
    MLP_CK(e);
    return NDSI_OK;
}

int ndsi_mlp_train(float* params, const float* X, const float* T, int32_t n, int32_t steps, float lr,
                   float* loss_out, void* stream) {
    if (!params || !X || !T || n < 1 || steps < 1 || !(lr > 0) || !dev_ptr(params) || !dev_ptr(X) || !dev_ptr(T))
        return mfail(NDSI_ERR_INVALID, "ndsi_mlp_train: device arrays, n >= 1, steps >= 1, lr > 0 required");
    static bool attr = false;
    if (!attr) {
        for (auto f : {&k_mlp_grad<true>, &k_mlp_grad<false>})
            MLP_CK(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(grad_smem())));
        attr = true;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int nblk = grad_blocks(n);
    float* work = nullptr;
    const size_t nwork = static_cast<size_t>(nblk) * kNParams + nblk + 2 * kNParams + 1;
    MLP_CK(cudaMalloc(&work, sizeof(float) * nwork));
    float* partial = work;
    float* lossp = partial + static_cast<size_t>(nblk) * kNParams;
    float* m = lossp + nblk;
    float* v = m + kNParams;
    float* loss = v + kNParams;
    cudaError_t e = cudaMemsetAsync(m, 0, sizeof(float) * 2 * kNParams, st);
    int rc = NDSI_OK;
    const float b1 = 0.9f, b2 = 0.999f;
    double p1 = 1.0, p2 = 1.0;
    for (int s = 0; s < steps && rc == NDSI_OK && e == cudaSuccess; ++s) {
        p1 *= b1;
        p2 *= b2;
        const AdamStep adam{params, m, v, lr, b1, b2, 1e-8f, static_cast<float>(1.0 - p1), static_cast<float>(1.0 - p2)};
        rc = grad_launch(params, X, T, n, partial, lossp, nullptr, loss, adam, st);
    }
    if (e == cudaSuccess && loss_out) e = cudaMemcpyAsync(loss_out, loss, sizeof(float), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(work);
    if (rc) return rc;
    MLP_CK(e);
    return NDSI_OK;
}

}  // extern "C"
