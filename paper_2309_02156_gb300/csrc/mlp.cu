// Learned coefficient predictor: a small MLP that predicts the history
// coefficients y of the guess from the coefficient vectors of the previous
// four systems and the sketched residual of the linearly extrapolated guess
// (the paper computes y by least squares every step, Algorithm 1; this
// is the learned variant, with the sketched least squares as fallback).
//
// Network: 4M+s -> H -> H -> M, GELU (erf form), weights stored FP32 (master)
// and rounded to bfloat16 (round to nearest even) for every forward and
// backward pass, FP32 arithmetic and accumulation.  Output head:
// y_hat = shift(y_{i-1}) + sigma_out * d.  Loss per sample:
// (y_hat - y)^T (W1^T W1) (y_hat - y) / ||wb||^2, the excess sketched residual
// over the least-squares minimum.  Adam (bias-corrected).  Every reduction
// (GEMM dot products, batch sums) runs in a fixed order: training is
// deterministic.
//
// Sample layout (FP32, stride in + out + out*out + 1):
//   [features (in) | target y (out) | G = W1^T W1 (out x out) | ||wb||].
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "../../include/seqaccel.h"
#include "common.cuh"
#include "internal.h"
#include "mlp_internal.h"

#include <cuda_bf16.h>

namespace sa {
namespace {

constexpr int TB = 16;   // GEMM tile

__device__ __forceinline__ float gelu_f(float u) { return 0.5f * u * (1.0f + erff(u * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_d(float u) {
    return 0.5f * (1.0f + erff(u * 0.70710678118654752f)) +
           u * expf(-0.5f * u * u) * 0.39894228040143268f;
}
__device__ __forceinline__ float bf(uint16_t v) {
    return __bfloat162float(__ushort_as_bfloat16(v));
}

// The GEMMs are tiny (at most 64 x 256 x 256 in use), so a kernel's time is the
// latency of its loads: each block loads kChunk of the summed index at once
// (16 before, one load latency and two barriers per 16 terms: 137 us per batch
// of 32, now 56 with the launches below).  Every output stays one chain of fused multiply-adds in the
// order of the summed index, zeros up to a multiple of 16 included, so results
// are the same bits as with the smaller tiles.
constexpr int kChunk = 128;
constexpr int kStride = kChunk + 1;

struct Tiles {
    float a[TB * kStride], b[TB * kStride];
};

// Rows of a batch: sample idx[r] of S (idx NULL: r).
__device__ __forceinline__ const float* sample_row(const float* S, int stride, const int* idx, int r) {
    return S + (size_t)(idx ? idx[r] : r) * stride;
}

// Y = X W^T + b (X: B x K fp32, W: N x K bf16); optional H = GELU(Y).
// FIRST: X is the normalised features of the samples, also written to z.
template <bool FIRST>
__global__ void __launch_bounds__(TB * TB)
linear_fwd(const float* __restrict__ X, int ldx, const uint16_t* __restrict__ W,
           const float* __restrict__ bias, int B, int N, int K, float* A, float* H,
           const int* __restrict__ idx, const float* __restrict__ mu, const float* __restrict__ sd,
           float* z) {
    __shared__ Tiles t;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TB + tx;
    const int row = blockIdx.y * TB + ty, col = blockIdx.x * TB + tx;
    float acc = 0.f;
    for (int k0 = 0; k0 < K; k0 += kChunk) {
#pragma unroll
        for (int q = 0; q < kChunk / TB; ++q) {
            const int i = tid + q * TB * TB, r = i / kChunk, k = i % kChunk;
            const int br = blockIdx.y * TB + r, wn = blockIdx.x * TB + r;
            float xv = 0.f;
            if (br < B && k0 + k < K) {
                if constexpr (FIRST) {
                    xv = (sample_row(X, ldx, idx, br)[k0 + k] - mu[k0 + k]) / sd[k0 + k];
                    if (blockIdx.x == 0) z[(size_t)br * K + k0 + k] = xv;
                } else {
                    xv = X[(size_t)br * ldx + k0 + k];
                }
            }
            t.a[r * kStride + k] = xv;
            t.b[r * kStride + k] = (wn < N && k0 + k < K) ? bf(W[(size_t)wn * K + k0 + k]) : 0.f;
        }
        __syncthreads();
        const int m = min(kChunk, (K - k0 + TB - 1) / TB * TB);
#pragma unroll 16
        for (int k = 0; k < m; ++k) acc = fmaf(t.a[ty * kStride + k], t.b[tx * kStride + k], acc);
        __syncthreads();
    }
    if (row < B && col < N) {
        const float a = acc + bias[col];
        A[(size_t)row * N + col] = a;
        if (H) H[(size_t)row * N + col] = gelu_f(a);
    }
}

// dX = (dY W) * GELU'(Apre)   (dY: B x N, W: N x K bf16, dX: B x K), block (bx, by).
__device__ void bwd_input_block(Tiles& t, int bx, int by, const float* __restrict__ dY,
                                const uint16_t* __restrict__ W, const float* __restrict__ Apre, int B,
                                int N, int K, float* dX) {
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TB + tx;
    const int row = by * TB + ty, col = bx * TB + tx;
    float acc = 0.f;
    for (int n0 = 0; n0 < N; n0 += kChunk) {
#pragma unroll
        for (int q = 0; q < kChunk / TB; ++q) {
            const int i = tid + q * TB * TB;
            const int r = i / kChunk, n = i % kChunk;            // dY: by rows
            t.a[r * kStride + n] = (by * TB + r < B && n0 + n < N) ? dY[(size_t)(by * TB + r) * N + n0 + n] : 0.f;
            const int wn = i / TB, wk = bx * TB + i % TB;        // W: TB columns of each row
            t.b[(i % TB) * kStride + wn] = (n0 + wn < N && wk < K) ? bf(W[(size_t)(n0 + wn) * K + wk]) : 0.f;
        }
        __syncthreads();
        const int m = min(kChunk, (N - n0 + TB - 1) / TB * TB);
#pragma unroll 16
        for (int n = 0; n < m; ++n) acc = fmaf(t.a[ty * kStride + n], t.b[tx * kStride + n], acc);
        __syncthreads();
    }
    if (row < B && col < K) {
        const float g = Apre ? gelu_d(Apre[(size_t)row * K + col]) : 1.f;
        dX[(size_t)row * K + col] = acc * g;
    }
}

// dW = dY^T X (N x K), db = sum_b dY (b in order), block (bx, by).
__device__ void bwd_weight_block(Tiles& t, int bx, int by, const float* __restrict__ dY,
                                 const float* __restrict__ X, int ldx, int B, int N, int K, float* dW,
                                 float* db) {
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TB + tx;
    const int n = by * TB + ty, k = bx * TB + tx;
    float acc = 0.f, bacc = 0.f;
    for (int b0 = 0; b0 < B; b0 += kChunk) {
#pragma unroll
        for (int q = 0; q < kChunk / TB; ++q) {
            const int i = tid + q * TB * TB, b = i / TB, c = i % TB;   // TB columns of each sample
            t.a[c * kStride + b] = (b0 + b < B && by * TB + c < N) ? dY[(size_t)(b0 + b) * N + by * TB + c] : 0.f;
            t.b[c * kStride + b] = (b0 + b < B && bx * TB + c < K) ? X[(size_t)(b0 + b) * ldx + bx * TB + c] : 0.f;
        }
        __syncthreads();
        const int m = min(kChunk, (B - b0 + TB - 1) / TB * TB);
#pragma unroll 16
        for (int b = 0; b < m; ++b) acc = fmaf(t.a[ty * kStride + b], t.b[tx * kStride + b], acc);
        if (bx == 0 && tx == 0)
            for (int b = 0; b < m; ++b) bacc += t.a[ty * kStride + b];
        __syncthreads();
    }
    if (n < N && k < K) dW[(size_t)n * K + k] = acc;
    if (bx == 0 && tx == 0 && n < N) db[n] = bacc;
}

// Both gradients of one layer in one launch (they share only dY): blocks
// [0, wx wy) form dW and db, the others dX (none when dX is NULL).  sum_out: block
// 0 also writes the mean of loss[0..B) (added in order).
__global__ void __launch_bounds__(TB * TB)
linear_bwd(const float* __restrict__ dY, const float* __restrict__ X, int ldx,
           const uint16_t* __restrict__ W, const float* __restrict__ Apre, int B, int N, int K,
           float* dW, float* db, float* dX, const float* __restrict__ loss, float* sum_out) {
    __shared__ Tiles t;
    const int wx = (K + TB - 1) / TB, wy = (N + TB - 1) / TB;
    const int blk = blockIdx.x;
    if (blk < wx * wy)
        bwd_weight_block(t, blk % wx, blk / wx, dY, X, ldx, B, N, K, dW, db);
    else
        bwd_input_block(t, (blk - wx * wy) % wx, (blk - wx * wy) / wx, dY, W, Apre, B, N, K, dX);
    if (sum_out && blk == 0 && threadIdx.x == 0 && threadIdx.y == 0) {
        float s = 0.f;
        for (int i = 0; i < B; ++i) s += loss[i];
        *sum_out = s / (float)B;
    }
}

// y = base + sigma * d; for training also the loss gradient and per-sample
// loss.  A warp per sample (one output per lane; out <= 31).
__global__ void __launch_bounds__(128)
head_kernel(const float* __restrict__ S, int stride, int B, int out, const float* __restrict__ d,
            const float* __restrict__ sig, int in, float* y, float* dd, float* loss,
            const int* __restrict__ idx) {
    __shared__ float es[4][32], gs[4][32];
    const int w = threadIdx.x >> 5, j = threadIdx.x & 31, b = blockIdx.x * 4 + w;
    if (b >= B) return;
    const float* s = sample_row(S, stride, idx, b);
    float yy = 0.f, e = 0.f;
    const float* T = s + in;
    if (j < out) {
        yy = s[j] + sig[j] * d[(size_t)b * out + j];
        if (y) y[(size_t)b * out + j] = yy;
        if (dd) e = yy - T[j];
    }
    if (!dd) return;
    es[w][j] = e;
    __syncwarp();
    const float* G = T + out;
    const float nb = s[in + out + out * out];
    const float inv = 1.f / (nb * nb);
    float ge = 0.f;
    if (j < out) {
        for (int k = 0; k < out; ++k) ge = fmaf(G[j * out + k], es[w][k], ge);
        dd[(size_t)b * out + j] = (2.f / (float)B) * ge * inv * sig[j];
    }
    gs[w][j] = ge;
    __syncwarp();
    if (j == 0) {
        float l = 0.f;
        for (int k = 0; k < out; ++k) l = fmaf(es[w][k], gs[w][k], l);
        loss[b] = l * inv;
    }
}

// Where the bf16 copy of parameter i lies: three weight blocks, biases have none.
struct Bf16Map {
    size_t at[3], end[3], to[3];
    uint16_t* W;
};

__global__ void adam_kernel(float* P, const float* __restrict__ G, float* M, float* V, size_t n,
                            float lr, float b1, float b2, float eps, float c1, float c2,
                            const Bf16Map map) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const float g = G[i];
        const float m = b1 * M[i] + (1.f - b1) * g;
        const float v = b2 * V[i] + (1.f - b2) * g * g;
        M[i] = m;
        V[i] = v;
        float p = P[i];
        p -= lr * (m / c1) / (sqrtf(v / c2) + eps);
        P[i] = p;
#pragma unroll
        for (int q = 0; q < 3; ++q)
            if (i >= map.at[q] && i < map.end[q])
                map.W[map.to[q] + (i - map.at[q])] = __bfloat16_as_ushort(__float2bfloat16_rn(p));
    }
}

__global__ void to_bf16_kernel(const float* __restrict__ P, uint16_t* W, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        W[i] = __bfloat16_as_ushort(__float2bfloat16_rn(P[i]));
}

// He-uniform weights from SplitMix64 outputs offset+1 .., biases zero.
__global__ void he_init_kernel(float* W, size_t n, int fan_in, uint64_t seed, uint64_t offset) {
    const double bound = sqrt(6.0 / (double)fan_in);
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const uint64_t h = mix64(seed + (offset + i + 1) * 0x9E3779B97F4A7C15ull);
        const double u = (double)(h >> 11) * (1.0 / 9007199254740992.0);
        W[i] = (float)((2.0 * u - 1.0) * bound);
    }
}

// Per-feature mean/std over the samples, and per-output std of (target - base).
__global__ void norm_stats_kernel(const float* __restrict__ S, int stride, int count, int in,
                                  int out, float* mu, float* sd, float* sig) {
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f < in) {
        double s = 0, s2 = 0;
        int b = 0;
        for (; b + 16 <= count; b += 16) {        // loads ahead of the ordered sums
            float v[16];
#pragma unroll
            for (int u = 0; u < 16; ++u) v[u] = S[(size_t)(b + u) * stride + f];
#pragma unroll
            for (int u = 0; u < 16; ++u) {
                const double w = v[u];
                s += w;
                s2 += w * w;
            }
        }
        for (; b < count; ++b) {
            const double v = S[(size_t)b * stride + f];
            s += v;
            s2 += v * v;
        }
        const double m = s / count, var = fmax(s2 / count - m * m, 0.0);
        mu[f] = (float)m;
        sd[f] = (float)fmax(sqrt(var), 1e-6);
    } else if (f < in + out) {
        const int j = f - in;
        double s2 = 0;
        int b = 0;
        for (; b + 16 <= count; b += 16) {
            float v[16];
#pragma unroll
            for (int u = 0; u < 16; ++u) v[u] = S[(size_t)(b + u) * stride + in + j] - S[(size_t)(b + u) * stride + j];
#pragma unroll
            for (int u = 0; u < 16; ++u) {
                const double w = v[u];
                s2 += w * w;
            }
        }
        for (; b < count; ++b) {
            const double v = S[(size_t)b * stride + in + j] - S[(size_t)b * stride + j];
            s2 += v * v;
        }
        sig[j] = (float)fmax(sqrt(s2 / count), 1e-6);
    }
}

}  // namespace

// ---- pieces used by the learned guess in api.cu ----------------------------

// Training sample of the current guess: features from the sketched block of
// the current window and the previous coefficient vectors (ring, newest
// first), target = the least-squares y, G = W1^T W1, ||wb||.
__global__ void learned_sample_kernel(const LsqOut* __restrict__ lo, int s, int M,
                                      const double* __restrict__ yring, float* sample) {
    __shared__ double Wl[kMaxS * (kMaxM + 1)];
    const int ncol = M + 1, in = 4 * M + s, tid = threadIdx.x;
    for (int i = tid; i < s * ncol; i += blockDim.x) Wl[i] = lo->W_logical[i];
    __syncthreads();
    __shared__ double nb;
    if (tid == 0) {
        double t = 0;
        for (int q = 0; q < s; ++q) t += Wl[q * ncol + M] * Wl[q * ncol + M];
        nb = sqrt(t);
    }
    __syncthreads();
    for (int k = 1; k <= 4; ++k)
        for (int j = tid; j < M; j += blockDim.x) {
            const int src = j + k;
            sample[(k - 1) * M + j] = src < M ? (float)yring[(k - 1) * kMaxM + src] : 0.f;
        }
    for (int q = tid; q < s; q += blockDim.x) {
        const double e = 2.0 * Wl[q * ncol + M - 1] - (M >= 2 ? Wl[q * ncol + M - 2] : 0.0) - Wl[q * ncol + M];
        sample[4 * M + q] = (float)(e / nb);
    }
    for (int j = tid; j < M; j += blockDim.x) sample[in + j] = (float)lo->y_logical[j];
    for (int jk = tid; jk < M * M; jk += blockDim.x) {
        const int j = jk / M, k = jk - j * M;
        double g = 0;
        for (int q = 0; q < s; ++q) g += Wl[q * ncol + j] * Wl[q * ncol + k];
        sample[in + M + jk] = (float)g;
    }
    if (tid == 0) sample[in + M + M * M] = (float)nb;
}

// Choose between the network's prediction and the least-squares solution:
// the network's y is used unless its sketched residual exceeds 1.5 times the
// least-squares one.  Writes the chosen y into lo (logical and physical).
__global__ void learned_select_kernel(LsqOut* lo, int s, int M, int oldest, const float* __restrict__ yhat,
                                      int* used_net, double* rho_net_out) {
    __shared__ double part[32];
    const int ncol = M + 1, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double acc = 0;
    for (int q = tid; q < s; q += blockDim.x) {
        double r = -lo->W_logical[q * ncol + M];
        for (int j = 0; j < M; ++j) r += lo->W_logical[q * ncol + j] * (double)yhat[j];
        acc += r * r;
    }
    acc = warp_sum(acc);
    if (lane == 0) part[warp] = acc;
    __syncthreads();
    __shared__ int use;
    if (tid == 0) {
        double t = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += part[w];
        const double rho_net = sqrt(t);
        use = rho_net <= 1.5 * lo->rho;
        *rho_net_out = rho_net;
        if (use) lo->rho = rho_net;
        *used_net = use;
    }
    __syncthreads();
    if (use) {
        for (int j = tid; j < M; j += blockDim.x) {
            lo->y_logical[j] = (double)yhat[j];
            lo->y_phys[(oldest + j) % M] = (double)yhat[j];
        }
    }
}

// Ring of the last four coefficient vectors (newest first), in the frame of
// the window they were computed for.
__global__ void yring_push_kernel(double* yring, const LsqOut* __restrict__ lo, int M) {
    const int j = threadIdx.x;
    if (j >= M) return;
    for (int k = 3; k >= 1; --k) yring[k * kMaxM + j] = yring[(k - 1) * kMaxM + j];
    yring[j] = lo->y_logical[j];
}

void launch_learned_sample(const LsqOut* lo, int s, int M, const double* yring, float* sample,
                           cudaStream_t st) {
    learned_sample_kernel<<<1, 256, 0, st>>>(lo, s, M, yring, sample);
}
void launch_learned_select(LsqOut* lo, int s, int M, int oldest, const float* yhat, int* used,
                           double* rho_net, cudaStream_t st) {
    learned_select_kernel<<<1, 128, 0, st>>>(lo, s, M, oldest, yhat, used, rho_net);
}
void launch_yring_push(double* yring, const LsqOut* lo, int M, cudaStream_t st) {
    yring_push_kernel<<<1, 32, 0, st>>>(yring, lo, M);
}

}  // namespace sa

using namespace sa;

struct seq_mlp {
    int M, s, in, hid, out, bmax, stride;
    cudaStream_t stream;
    size_t oW1, ob1, oW2, ob2, oW3, ob3, np;
    float *P = nullptr, *G = nullptr, *Mm = nullptr, *Vv = nullptr;
    uint16_t* Wb = nullptr;            // bf16 W1 | W2 | W3
    float *mu = nullptr, *sd = nullptr, *sig = nullptr;
    float *z, *a1, *h1, *a2, *h2, *d, *y, *dd, *dh2, *dh1, *loss, *scalar;
    int* idx = nullptr;                // a training call's batches, and its losses
    float* step_loss = nullptr;
    size_t idx_cap = 0, loss_cap = 0;
    int t = 0;
    std::vector<void*> allocs;
};

namespace {

int mlp_alloc(seq_mlp* m, void** p, size_t bytes) {
    if (cudaMalloc(p, bytes ? bytes : 4) != cudaSuccess) {
        cudaGetLastError();
        return SEQ_ENOMEM;
    }
    m->allocs.push_back(*p);
    return SEQ_OK;
}

// A buffer that grows and is kept for the next call.
int mlp_reserve(void** p, size_t* cap, size_t want, size_t size) {
    if (want <= *cap) return SEQ_OK;
    if (*p) cudaFree(*p);
    *p = nullptr;
    *cap = 0;
    if (cudaMalloc(p, size * want) != cudaSuccess) {
        cudaGetLastError();
        return SEQ_ENOMEM;
    }
    *cap = want;
    return SEQ_OK;
}

void refresh_bf16(seq_mlp* m) {
    const size_t n1 = (size_t)m->hid * m->in, n2 = (size_t)m->hid * m->hid, n3 = (size_t)m->out * m->hid;
    to_bf16_kernel<<<64, 256, 0, m->stream>>>(m->P + m->oW1, m->Wb, n1);
    to_bf16_kernel<<<64, 256, 0, m->stream>>>(m->P + m->oW2, m->Wb + n1, n2);
    to_bf16_kernel<<<16, 256, 0, m->stream>>>(m->P + m->oW3, m->Wb + n1 + n2, n3);
}

// Forward pass on B samples (rows idx[..] of S with the sample stride).
void mlp_forward(seq_mlp* m, const float* S, int stride, int B, cudaStream_t st,
                 const int* idx = nullptr) {
    const size_t n1 = (size_t)m->hid * m->in, n2 = (size_t)m->hid * m->hid;
    const dim3 blk(TB, TB), hidden((m->hid + TB - 1) / TB, (B + TB - 1) / TB);
    linear_fwd<true><<<hidden, blk, 0, st>>>(S, stride, m->Wb, m->P + m->ob1, B, m->hid, m->in, m->a1,
                                             m->h1, idx, m->mu, m->sd, m->z);
    linear_fwd<false><<<hidden, blk, 0, st>>>(m->h1, m->hid, m->Wb + n1, m->P + m->ob2, B, m->hid,
                                              m->hid, m->a2, m->h2, nullptr, nullptr, nullptr, nullptr);
    linear_fwd<false><<<dim3((m->out + TB - 1) / TB, (B + TB - 1) / TB), blk, 0, st>>>(
        m->h2, m->hid, m->Wb + n1 + n2, m->P + m->ob3, B, m->out, m->hid, m->d, nullptr, nullptr,
        nullptr, nullptr, nullptr);
}

// Loss (mean over the samples, to *mean) and gradients (into m->G) on B samples.
void mlp_backward(seq_mlp* m, const float* S, int stride, int B, const int* idx, float* mean) {
    const size_t n1 = (size_t)m->hid * m->in, n2 = (size_t)m->hid * m->hid;
    head_kernel<<<(B + 3) / 4, 128, 0, m->stream>>>(S, stride, B, m->out, m->d, m->sig, m->in, m->y,
                                                    m->dd, m->loss, idx);
    const dim3 blk(TB, TB);
    auto tiles = [](int n) { return (n + TB - 1) / TB; };
    const int bx = tiles(B);
    linear_bwd<<<tiles(m->hid) * (tiles(m->out) + bx), blk, 0, m->stream>>>(
        m->dd, m->h2, m->hid, m->Wb + n1 + n2, m->a2, B, m->out, m->hid, m->G + m->oW3, m->G + m->ob3,
        m->dh2, m->loss, mean);
    linear_bwd<<<tiles(m->hid) * (tiles(m->hid) + bx), blk, 0, m->stream>>>(
        m->dh2, m->h1, m->hid, m->Wb + n1, m->a1, B, m->hid, m->hid, m->G + m->oW2, m->G + m->ob2,
        m->dh1, nullptr, nullptr);
    linear_bwd<<<tiles(m->in) * tiles(m->hid), blk, 0, m->stream>>>(
        m->dh1, m->z, m->in, nullptr, nullptr, B, m->hid, m->in, m->G + m->oW1, m->G + m->ob1, nullptr,
        nullptr, nullptr);
}

}  // namespace

namespace sa {
// Prediction on stream st (the predictor's activations are reused: not
// concurrently with training on another stream).
void mlp_predict_dev(seq_mlp* m, const float* features, int B, float* y, cudaStream_t st) {
    mlp_forward(m, features, m->stride, B, st);
    head_kernel<<<(B + 3) / 4, 128, 0, st>>>(features, m->stride, B, m->out, m->d, m->sig, m->in, y,
                                             nullptr, nullptr, nullptr);
}
int mlp_stride(const seq_mlp* m) { return m->stride; }
int mlp_dims_ok(const seq_mlp* m, int M, int s) { return m && m->M == M && m->s == s; }
int mlp_hidden(const seq_mlp* m) { return m ? m->hid : 0; }
int mlp_max_batch(const seq_mlp* m) { return m ? m->bmax : 0; }
}  // namespace sa

extern "C" {

int seq_mlp_create(int32_t M, int32_t s, int32_t hidden, int32_t max_batch, uint64_t seed,
                   void* cuda_stream, seq_mlp** out) {
    if (!out) return SEQ_EINVAL;
    *out = nullptr;
    if (M < 2 || M > kMaxM || s < M + 1 || s > kMaxS || hidden < 1 || hidden > 4096 ||
        max_batch < 1 || max_batch > 65536)
        return SEQ_EINVAL;
    seq_mlp* m = new seq_mlp();
    m->M = M;
    m->s = s;
    m->in = 4 * M + s;
    m->hid = hidden;
    m->out = M;
    m->bmax = max_batch;
    m->stride = m->in + M + M * M + 1;
    m->stream = (cudaStream_t)cuda_stream;
    m->oW1 = 0;
    m->ob1 = m->oW1 + (size_t)m->hid * m->in;
    m->oW2 = m->ob1 + m->hid;
    m->ob2 = m->oW2 + (size_t)m->hid * m->hid;
    m->oW3 = m->ob2 + m->hid;
    m->ob3 = m->oW3 + (size_t)m->out * m->hid;
    m->np = m->ob3 + m->out;
    int rc = SEQ_OK;
    void* p;
    auto A = [&](float** dst, size_t nfl) {
        if (rc == SEQ_OK) {
            rc = mlp_alloc(m, &p, nfl * sizeof(float));
            *dst = (float*)p;
        }
    };
    A(&m->P, m->np);
    A(&m->G, m->np);
    A(&m->Mm, m->np);
    A(&m->Vv, m->np);
    A(&m->mu, m->in);
    A(&m->sd, m->in);
    A(&m->sig, m->out);
    const size_t B = m->bmax;
    A(&m->z, B * m->in);
    A(&m->a1, B * m->hid);
    A(&m->h1, B * m->hid);
    A(&m->a2, B * m->hid);
    A(&m->h2, B * m->hid);
    A(&m->d, B * m->out);
    A(&m->y, B * m->out);
    A(&m->dd, B * m->out);
    A(&m->dh2, B * m->hid);
    A(&m->dh1, B * m->hid);
    A(&m->loss, B);
    A(&m->scalar, 4);
    if (rc == SEQ_OK) {
        rc = mlp_alloc(m, &p, sizeof(uint16_t) * ((size_t)m->hid * m->in + (size_t)m->hid * m->hid +
                                                   (size_t)m->out * m->hid));
        m->Wb = (uint16_t*)p;
    }
    if (rc != SEQ_OK) {
        seq_mlp_destroy(m);
        return rc;
    }
    cudaMemsetAsync(m->P, 0, sizeof(float) * m->np, m->stream);
    cudaMemsetAsync(m->Mm, 0, sizeof(float) * m->np, m->stream);
    cudaMemsetAsync(m->Vv, 0, sizeof(float) * m->np, m->stream);
    he_init_kernel<<<64, 256, 0, m->stream>>>(m->P + m->oW1, (size_t)m->hid * m->in, m->in, seed, 0);
    he_init_kernel<<<64, 256, 0, m->stream>>>(m->P + m->oW2, (size_t)m->hid * m->hid, m->hid, seed,
                                              (uint64_t)m->hid * m->in);
    he_init_kernel<<<16, 256, 0, m->stream>>>(m->P + m->oW3, (size_t)m->out * m->hid, m->hid, seed,
                                              (uint64_t)m->hid * m->in + (uint64_t)m->hid * m->hid);
    std::vector<float> ones(m->in, 1.f);
    cudaMemsetAsync(m->mu, 0, sizeof(float) * m->in, m->stream);
    cudaMemcpy(m->sd, ones.data(), sizeof(float) * m->in, cudaMemcpyHostToDevice);
    cudaMemcpy(m->sig, ones.data(), sizeof(float) * m->out, cudaMemcpyHostToDevice);
    refresh_bf16(m);
    if (cudaStreamSynchronize(m->stream) != cudaSuccess || cudaGetLastError() != cudaSuccess) {
        seq_mlp_destroy(m);
        return SEQ_ECUDA;
    }
    *out = m;
    return SEQ_OK;
}

int seq_mlp_destroy(seq_mlp* m) {
    if (!m) return SEQ_OK;
    cudaStreamSynchronize(m->stream);
    for (void* p : m->allocs) cudaFree(p);
    if (m->idx) cudaFree(m->idx);
    if (m->step_loss) cudaFree(m->step_loss);
    delete m;
    return SEQ_OK;
}

int seq_mlp_param_count(const seq_mlp* m) { return m ? (int)m->np : 0; }

int seq_mlp_get_params(seq_mlp* m, float* params_host, float* norm_host) {
    if (!m) return SEQ_EINVAL;
    if (cudaStreamSynchronize(m->stream) != cudaSuccess) return SEQ_ECUDA;
    if (params_host && cudaMemcpy(params_host, m->P, sizeof(float) * m->np, cudaMemcpyDeviceToHost) != cudaSuccess)
        return SEQ_ECUDA;
    if (norm_host) {
        if (cudaMemcpy(norm_host, m->mu, sizeof(float) * m->in, cudaMemcpyDeviceToHost) != cudaSuccess ||
            cudaMemcpy(norm_host + m->in, m->sd, sizeof(float) * m->in, cudaMemcpyDeviceToHost) != cudaSuccess ||
            cudaMemcpy(norm_host + 2 * m->in, m->sig, sizeof(float) * m->out, cudaMemcpyDeviceToHost) != cudaSuccess)
            return SEQ_ECUDA;
    }
    return SEQ_OK;
}

int seq_mlp_set_params(seq_mlp* m, const float* params_host, const float* norm_host) {
    if (!m) return SEQ_EINVAL;
    if (params_host && cudaMemcpyAsync(m->P, params_host, sizeof(float) * m->np, cudaMemcpyHostToDevice,
                                       m->stream) != cudaSuccess)
        return SEQ_ECUDA;
    if (norm_host) {
        cudaMemcpyAsync(m->mu, norm_host, sizeof(float) * m->in, cudaMemcpyHostToDevice, m->stream);
        cudaMemcpyAsync(m->sd, norm_host + m->in, sizeof(float) * m->in, cudaMemcpyHostToDevice, m->stream);
        cudaMemcpyAsync(m->sig, norm_host + 2 * m->in, sizeof(float) * m->out, cudaMemcpyHostToDevice, m->stream);
    }
    refresh_bf16(m);
    m->t = 0;
    cudaMemsetAsync(m->Mm, 0, sizeof(float) * m->np, m->stream);
    cudaMemsetAsync(m->Vv, 0, sizeof(float) * m->np, m->stream);
    return cudaStreamSynchronize(m->stream) == cudaSuccess ? SEQ_OK : SEQ_ECUDA;
}

int seq_mlp_fit_normalization(seq_mlp* m, const float* samples_dev, int32_t count) {
    if (!m || !samples_dev || count < 1) return SEQ_EINVAL;
    norm_stats_kernel<<<(m->in + m->out + 127) / 128, 128, 0, m->stream>>>(samples_dev, m->stride, count,
                                                                          m->in, m->out, m->mu, m->sd, m->sig);
    return cudaStreamSynchronize(m->stream) == cudaSuccess ? SEQ_OK : SEQ_ECUDA;
}

int seq_mlp_loss_grad(seq_mlp* m, const float* samples_dev, int32_t B, float* loss_host,
                      float* grads_host) {
    if (!m || !samples_dev || B < 1 || B > m->bmax) return SEQ_EINVAL;
    mlp_forward(m, samples_dev, m->stride, B, m->stream);
    mlp_backward(m, samples_dev, m->stride, B, nullptr, m->scalar);
    if (cudaStreamSynchronize(m->stream) != cudaSuccess) return SEQ_ECUDA;
    if (loss_host && cudaMemcpy(loss_host, m->scalar, sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess)
        return SEQ_ECUDA;
    if (grads_host && cudaMemcpy(grads_host, m->G, sizeof(float) * m->np, cudaMemcpyDeviceToHost) != cudaSuccess)
        return SEQ_ECUDA;
    return SEQ_OK;
}

int seq_mlp_train(seq_mlp* m, const float* samples_dev, int32_t count, int32_t epochs, int32_t batch,
                  float lr, uint64_t seed, float* losses_host) {
    if (!m || !samples_dev || count < 1 || epochs < 0 || batch < 1 || batch > m->bmax || !(lr > 0))
        return SEQ_EINVAL;
    // The sample numbers of as many epochs as kMaxRows allows go up at once and
    // their batches' losses come back together: one synchronisation per group.
    constexpr long long kMaxRows = 1 << 22;
    const int nb = count / batch;
    const long long per_epoch = (long long)nb * batch;
    const int group = per_epoch > 0 ? (int)std::max(1LL, std::min((long long)epochs, kMaxRows / per_epoch)) : 1;
    std::vector<int> perm(count), rows;
    std::vector<float> losses, ep_loss(epochs > 0 ? epochs : 1, 0.f);
    Bf16Map map;
    const size_t at[3] = {m->oW1, m->oW2, m->oW3};
    const size_t len[3] = {(size_t)m->hid * m->in, (size_t)m->hid * m->hid, (size_t)m->out * m->hid};
    map.W = m->Wb;
    for (size_t q = 0, to = 0; q < 3; to += len[q], ++q) {
        map.at[q] = at[q];
        map.end[q] = at[q] + len[q];
        map.to[q] = to;
    }
    uint64_t ctr = 0;
    for (int e0 = 0; e0 < epochs && nb > 0; e0 += group) {
        const int ne = std::min(group, epochs - e0);
        const size_t steps = (size_t)ne * nb;
        rows.clear();
        for (int e = 0; e < ne; ++e) {
            for (int i = 0; i < count; ++i) perm[i] = i;
            for (int i = count - 1; i > 0; --i) {      // Fisher-Yates with SplitMix64 draws
                uint64_t z = seed + (++ctr) * 0x9E3779B97F4A7C15ull;
                z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
                z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
                z ^= z >> 31;
                const int j = (int)(((z >> 32) * (uint64_t)(i + 1)) >> 32);
                std::swap(perm[i], perm[j]);
            }
            rows.insert(rows.end(), perm.begin(), perm.begin() + per_epoch);
        }
        losses.resize(steps);
        int rc = mlp_reserve((void**)&m->idx, &m->idx_cap, rows.size(), sizeof(int));
        if (!rc) rc = mlp_reserve((void**)&m->step_loss, &m->loss_cap, steps, sizeof(float));
        if (rc) return rc;
        if (cudaMemcpyAsync(m->idx, rows.data(), sizeof(int) * rows.size(), cudaMemcpyHostToDevice,
                            m->stream) != cudaSuccess)
            return SEQ_ECUDA;
        for (size_t i = 0; i < steps; ++i) {
            const int* idx = m->idx + i * batch;
            mlp_forward(m, samples_dev, m->stride, batch, m->stream, idx);
            mlp_backward(m, samples_dev, m->stride, batch, idx, m->step_loss + i);
            m->t += 1;
            const float c1 = 1.f - powf(0.9f, (float)m->t), c2 = 1.f - powf(0.999f, (float)m->t);
            adam_kernel<<<256, 256, 0, m->stream>>>(m->P, m->G, m->Mm, m->Vv, m->np, lr, 0.9f, 0.999f,
                                                    1e-8f, c1, c2, map);
        }
        if (cudaMemcpyAsync(losses.data(), m->step_loss, sizeof(float) * steps, cudaMemcpyDeviceToHost,
                            m->stream) != cudaSuccess ||
            cudaStreamSynchronize(m->stream) != cudaSuccess)
            return SEQ_ECUDA;
        for (int e = 0; e < ne; ++e) {
            double acc = 0;
            for (int i = 0; i < nb; ++i) acc += losses[(size_t)e * nb + i];
            ep_loss[e0 + e] = (float)(acc / nb);
        }
    }
    if (losses_host && epochs > 0) memcpy(losses_host, ep_loss.data(), sizeof(float) * epochs);
    return cudaGetLastError() == cudaSuccess ? SEQ_OK : SEQ_ECUDA;
}

int seq_mlp_predict(seq_mlp* m, const float* samples_dev, int32_t B, float* y_dev) {
    if (!m || !samples_dev || !y_dev || B < 1 || B > m->bmax) return SEQ_EINVAL;
    mlp_predict_dev(m, samples_dev, B, y_dev, m->stream);
    return cudaStreamSynchronize(m->stream) == cudaSuccess ? SEQ_OK : SEQ_ECUDA;
}

}  // extern "C"
