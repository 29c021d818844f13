// The cost model's network: 3-layer tanh perceptron, FP32, with hand-written
// forward, backward and Adam kernels (see tsm_mlp.h for the maths and the
// parameter layout).
//
// A call is a few hundred MFLOP at most (6126 samples, 17-64-64-1: 0.18
// GFLOP, 2.6 us at the FP32 rate), so what bounds it is latency: how many
// threads share the work, and how long the serial chains are.  Forward and
// gradient run as one kernel over tiles of 32 samples whose weights and
// activations stay in shared memory; each thread owns a small register tile
// of every layer product (2 samples x 4 units forward, 4 x 4 weights
// backward), and the CTA adds up its samples' share of the gradient in
// registers.  A second kernel sums the CTA shares.  Every order is fixed, so
// results repeat bit for bit, and each activation is the same ascending FMA
// chain as one thread per sample would run.
// Measured (6126 samples, D = 17, H = 64, loss and gradient with its copy to
// the host): 1415 us with one thread per sample and one per parameter over
// all samples (a chain of 6126 dependent FMAs), 58 us now.
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "tsm_internal.h"
#include "tsm_mlp.h"

struct tsm_mlp {
    int D, H, max_batch, P;
    float* params;  // device
    float* grads;
    float* m;
    float* v;
    float* parts;   // kMaxGrid x P: the CTAs' shares of the gradient
    double* lparts; // kMaxGrid: their shares of the squared error
    int grid_max;   // CTAs the shares are sized for
    int64_t step;
};

namespace tsm {
namespace mlp {

struct Off {
    int W1, b1, W2, b2, w3, b3, P;
};
__host__ __device__ inline Off offsets(int D, int H) {
    Off o;
    o.W1 = 0;
    o.b1 = H * D;
    o.W2 = o.b1 + H;
    o.b2 = o.W2 + H * H;
    o.w3 = o.b2 + H;
    o.b3 = o.w3 + H;
    o.P = o.b3 + 1;
    return o;
}

constexpr int kThreads = 256;
constexpr int TS = 32;              // samples per tile
constexpr int HMAX = TSM_MLP_MAX_HIDDEN, DMAX = TSM_MLP_MAX_IN;
constexpr int HS = HMAX + 4;        // row strides in floats: 16-byte aligned, and eight
constexpr int DS = DMAX + 4;        // consecutive rows fall into different banks
constexpr int kCtasPerSm = 2;       // CTAs of the gradient kernel per SM (85 KB of shared memory each)

// Shared memory of one CTA.  Rows and columns past H, D and the tile's
// samples hold zeros.
struct Smem {
    float W1[HMAX][DS], W2[HMAX][HS];
    float b1[HMAX], b2[HMAX], w3[HMAX];
    float x[TS][DS], h1[TS][HS], h2[TS][HS];
    float t[TS], dy[TS], y[TS];
    // gradient only
    float W2T[HMAX][HS], d1[TS][HS], d2[TS][HS];
};

// out[a][b] += sum over k < n4 (a multiple of 4) of X[s + 16a][k] W[u + 16b][k],
// k ascending: two LDS.128 of samples (broadcast) and four of weights feed
// 32 FMAs.
template <int XS, int WS>
__device__ __forceinline__ void layer(const float (*X)[XS], const float (*W)[WS], int n4, int s, int u,
                                      float (&out)[2][4]) {
    for (int k = 0; k < n4; k += 4) {
        float4 xv[2], wv[4];
#pragma unroll
        for (int a = 0; a < 2; ++a) xv[a] = *reinterpret_cast<const float4*>(&X[s + 16 * a][k]);
#pragma unroll
        for (int b = 0; b < 4; ++b) wv[b] = *reinterpret_cast<const float4*>(&W[u + 16 * b][k]);
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                out[a][b] = fmaf(wv[b].x, xv[a].x, out[a][b]);
                out[a][b] = fmaf(wv[b].y, xv[a].y, out[a][b]);
                out[a][b] = fmaf(wv[b].z, xv[a].z, out[a][b]);
                out[a][b] = fmaf(wv[b].w, xv[a].w, out[a][b]);
            }
    }
}

// GRAD = false: y[i] of every sample.  GRAD = true: this CTA's share of the
// gradient (parts + blockIdx.x * P) and of the squared error.  CTA b takes
// tiles b, b + gridDim.x, ...
template <bool GRAD>
__global__ void __launch_bounds__(kThreads) k_mlp(const float* __restrict__ p, int D, int H,
                                                  const float* __restrict__ X, const float* __restrict__ target,
                                                  int n, float* __restrict__ y, float* __restrict__ parts,
                                                  double* __restrict__ lparts) {
    extern __shared__ __align__(16) unsigned char raw[];
    Smem& S = *reinterpret_cast<Smem*>(raw);
    const Off o = offsets(D, H);
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int H4 = (H + 3) & ~3, D4 = (D + 3) & ~3;
    for (int i = tid; i < HMAX * DMAX; i += kThreads) {
        const int j = i / DMAX, k = i - j * DMAX;
        S.W1[j][k] = j < H && k < D ? p[o.W1 + j * D + k] : 0.0f;
    }
    for (int i = tid; i < HMAX * HMAX; i += kThreads) {
        const int j = i / HMAX, k = i - j * HMAX;
        const float w = j < H && k < H ? p[o.W2 + j * H + k] : 0.0f;
        S.W2[j][k] = w;
        if (GRAD) S.W2T[k][j] = w;
    }
    if (tid < HMAX) {
        S.b1[tid] = tid < H ? p[o.b1 + tid] : 0.0f;
        S.b2[tid] = tid < H ? p[o.b2 + tid] : 0.0f;
        S.w3[tid] = tid < H ? p[o.w3 + tid] : 0.0f;
    }
    const float b3 = p[o.b3];
    // gradient sums of this thread: W2[4ty + r][4tx + c], W1[4ty + r][tx + 16c],
    // and one entry of b1, b2, w3 or b3 (by thread index, below)
    float gW2[4][4] = {}, gW1[4][2] = {}, gv = 0.0f;
    double lsum = 0.0;
    const int tiles = (n + TS - 1) / TS;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int i0 = tile * TS, cnt = min(TS, n - i0);
        __syncthreads();  // weights staged; the previous tile is done with
        for (int i = tid; i < TS * DMAX; i += kThreads) {
            const int s = i / DMAX, k = i - s * DMAX;
            S.x[s][k] = s < cnt && k < D ? X[(int64_t)(i0 + s) * D + k] : 0.0f;
        }
        if (GRAD && tid < TS) S.t[tid] = tid < cnt ? target[i0 + tid] : 0.0f;
        __syncthreads();
        // units j >= H are set to zero, not computed: whatever the weights
        // hold, the padding stays zero
        float v[2][4];
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) v[a][b] = S.b1[tx + 16 * b];
        layer(S.x, S.W1, D4, ty, tx, v);
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) S.h1[ty + 16 * a][tx + 16 * b] = tx + 16 * b < H ? tanhf(v[a][b]) : 0.0f;
        __syncthreads();
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) v[a][b] = S.b2[tx + 16 * b];
        layer(S.h1, S.W2, H4, ty, tx, v);
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) S.h2[ty + 16 * a][tx + 16 * b] = tx + 16 * b < H ? tanhf(v[a][b]) : 0.0f;
        __syncthreads();
        if (tid < TS) {
            float s = b3;
            for (int k = 0; k < H; ++k) s = fmaf(S.w3[k], S.h2[tid][k], s);
            if (!GRAD) {
                if (tid < cnt) y[i0 + tid] = s;
            } else {
                const float e = tid < cnt ? s - S.t[tid] : 0.0f;
                S.y[tid] = e * e;
                S.dy[tid] = 2.0f * e / (float)n;
            }
        }
        if (!GRAD) continue;
        __syncthreads();
        // dL/d(pre-activation of layer 2)
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int s = ty + 16 * a, j = tx + 16 * b;
                const float h = S.h2[s][j];
                S.d2[s][j] = S.dy[s] * S.w3[j] * (1.0f - h * h);
                v[a][b] = 0.0f;
            }
        __syncthreads();
        // ... and of layer 1: sum over j of W2[j][k] dh2[j], j ascending
        layer(S.d2, S.W2T, H4, ty, tx, v);
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int s = ty + 16 * a, k = tx + 16 * b;
                const float h = S.h1[s][k];
                S.d1[s][k] = v[a][b] * (1.0f - h * h);
            }
        __syncthreads();
        // the tile's samples added to this thread's gradient entries
#pragma unroll 4
        for (int s = 0; s < cnt; ++s) {
            const float4 d = *reinterpret_cast<const float4*>(&S.d2[s][4 * ty]);
            const float4 h = *reinterpret_cast<const float4*>(&S.h1[s][4 * tx]);
            const float4 e = *reinterpret_cast<const float4*>(&S.d1[s][4 * ty]);
            const float x0 = S.x[s][tx], x1 = S.x[s][tx + 16];
            const float dv[4] = {d.x, d.y, d.z, d.w}, hv[4] = {h.x, h.y, h.z, h.w}, ev[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
            for (int r = 0; r < 4; ++r) {
#pragma unroll
                for (int c = 0; c < 4; ++c) gW2[r][c] = fmaf(dv[r], hv[c], gW2[r][c]);
                gW1[r][0] = fmaf(ev[r], x0, gW1[r][0]);
                gW1[r][1] = fmaf(ev[r], x1, gW1[r][1]);
            }
        }
        const int q = tid >> 6, j = tid & 63;
        if (q < 3) {
            for (int s = 0; s < cnt; ++s) {
                if (q == 0) gv += S.d1[s][j];
                if (q == 1) gv += S.d2[s][j];
                if (q == 2) gv = fmaf(S.dy[s], S.h2[s][j], gv);
            }
        } else if (j == 0) {
            for (int s = 0; s < cnt; ++s) gv += S.dy[s];
        } else if (j >= 32) {
            lsum += S.y[j - 32];  // one sample a lane; zero past the tile's samples
        }
    }
    if (!GRAD) return;
    float* g = parts + (int64_t)blockIdx.x * o.P;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int j = 4 * ty + r;
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (j < H && 4 * tx + c < H) g[o.W2 + j * H + 4 * tx + c] = gW2[r][c];
#pragma unroll
        for (int c = 0; c < 2; ++c)
            if (j < H && tx + 16 * c < D) g[o.W1 + j * D + tx + 16 * c] = gW1[r][c];
    }
    const int q = tid >> 6, j = tid & 63;
    if (q < 3) {
        if (j < H) g[(q == 0 ? o.b1 : (q == 1 ? o.b2 : o.w3)) + j] = gv;
    } else if (j == 0) {
        g[o.b3] = gv;
    } else if (j >= 32) {
#pragma unroll
        for (int h = 16; h >= 1; h >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, h);
        if (j == 32) lparts[blockIdx.x] = lsum;
    }
}

// Gradient and loss from the CTAs' shares.  Eight threads share a
// parameter (thread row r takes shares r, r + 8, ... in order), and the
// eight sums are combined by a fixed-pairing tree; the last CTA does the
// same for the loss, in double.
constexpr int kSlices = 8;
__global__ void __launch_bounds__(32 * kSlices) k_mlp_sum(const float* __restrict__ parts,
                                                          const double* __restrict__ lparts, int G, int P, int n,
                                                          float* __restrict__ g, float* __restrict__ loss) {
    __shared__ double red[kSlices][32];
    const int c = threadIdx.x & 31, r = threadIdx.x >> 5;
    if (blockIdx.x == gridDim.x - 1) {
        const int t = threadIdx.x;
        double s = 0.0;
        for (int b = t; b < G; b += 32 * kSlices) s += lparts[b];
        red[r][c] = s;
        __syncthreads();
        for (int h = 16 * kSlices; h >= 1; h >>= 1) {
            if (t < h) (&red[0][0])[t] += (&red[0][0])[t + h];
            __syncthreads();
        }
        if (t == 0) *loss = (float)(red[0][0] / n);
        return;
    }
    float* fr = reinterpret_cast<float*>(&red[0][0]);
    const int q = blockIdx.x * 32 + c;
    float s = 0.0f;
    if (q < P) {
#pragma unroll 8
        for (int b = r; b < G; b += kSlices) s += parts[(int64_t)b * P + q];
    }
    fr[r * 32 + c] = s;
    __syncthreads();
    for (int h = kSlices / 2; h >= 1; h >>= 1) {
        if (r < h) fr[r * 32 + c] += fr[(r + h) * 32 + c];
        __syncthreads();
    }
    if (r == 0 && q < P) g[q] = fr[c];
}

__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, int P, float lr, float b1, float b2, float eps, float c1, float c2) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= P) return;
    const float gq = g[q];
    const float mq = b1 * m[q] + (1.0f - b1) * gq;
    const float vq = b2 * v[q] + (1.0f - b2) * gq * gq;
    m[q] = mq;
    v[q] = vq;
    p[q] -= lr * (mq / c1) / (sqrtf(vq / c2) + eps);
}

uint64_t splitmix(uint64_t& s) {
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

}  // namespace mlp
}  // namespace tsm

using namespace tsm;

extern "C" {

tsm_status tsm_mlp_create(int in_dim, int hidden, int max_batch, uint64_t seed, tsm_mlp** out) {
    if (!out || in_dim < 1 || in_dim > TSM_MLP_MAX_IN || hidden < 1 || hidden > TSM_MLP_MAX_HIDDEN ||
        max_batch < 1)
        return TSM_ERR_INVALID_VALUE;
    *out = nullptr;
    tsm_mlp* m = (tsm_mlp*)calloc(1, sizeof(tsm_mlp));
    if (!m) return TSM_ERR_ALLOC;
    const mlp::Off o = mlp::offsets(in_dim, hidden);
    m->D = in_dim;
    m->H = hidden;
    m->max_batch = max_batch;
    m->P = o.P;
    const size_t pb = sizeof(float) * o.P;
    // one share per CTA: a resident wave, or fewer tiles than that
    const int sms = device_info().sm_count;
    m->grid_max = std::max(1, std::min((max_batch - 1) / mlp::TS + 1, mlp::kCtasPerSm * sms));
    bool ok = cudaMalloc(&m->params, pb) == cudaSuccess && cudaMalloc(&m->grads, pb) == cudaSuccess &&
              cudaMalloc(&m->m, pb) == cudaSuccess && cudaMalloc(&m->v, pb) == cudaSuccess &&
              cudaMalloc(&m->parts, pb * m->grid_max) == cudaSuccess &&
              cudaMalloc(&m->lparts, sizeof(double) * m->grid_max) == cudaSuccess;
    if (!ok) {
        tsm_mlp_destroy(m);
        return TSM_ERR_ALLOC;
    }
    std::vector<float> h(o.P, 0.0f);
    uint64_t s = seed;
    auto uni = [&](float bound) {
        return (float)(((double)(mlp::splitmix(s) >> 11) * 0x1p-53 * 2.0 - 1.0) * bound);
    };
    for (int i = 0; i < hidden * in_dim; ++i) h[o.W1 + i] = uni(1.0f / sqrtf((float)in_dim));
    for (int i = 0; i < hidden * hidden; ++i) h[o.W2 + i] = uni(1.0f / sqrtf((float)hidden));
    for (int i = 0; i < hidden; ++i) h[o.w3 + i] = uni(1.0f / sqrtf((float)hidden));
    if (cudaMemcpy(m->params, h.data(), pb, cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(m->grads, 0, pb) != cudaSuccess || cudaMemset(m->m, 0, pb) != cudaSuccess ||
        cudaMemset(m->v, 0, pb) != cudaSuccess) {
        tsm_mlp_destroy(m);
        return TSM_ERR_LAUNCH;
    }
    *out = m;
    return TSM_OK;
}

void tsm_mlp_destroy(tsm_mlp* m) {
    if (!m) return;
    cudaFree(m->params);
    cudaFree(m->grads);
    cudaFree(m->m);
    cudaFree(m->v);
    cudaFree(m->parts);
    cudaFree(m->lparts);
    free(m);
}

int tsm_mlp_param_count(const tsm_mlp* m) { return m ? m->P : -1; }

tsm_status tsm_mlp_set_params(tsm_mlp* m, const float* host) {
    if (!m || !host) return TSM_ERR_INVALID_VALUE;
    if (cudaMemcpy(m->params, host, sizeof(float) * m->P, cudaMemcpyHostToDevice) != cudaSuccess)
        return TSM_ERR_LAUNCH;
    // a new parameter vector restarts the optimiser
    if (cudaMemset(m->m, 0, sizeof(float) * m->P) != cudaSuccess ||
        cudaMemset(m->v, 0, sizeof(float) * m->P) != cudaSuccess)
        return TSM_ERR_LAUNCH;
    m->step = 0;
    return TSM_OK;
}

tsm_status tsm_mlp_get_params(const tsm_mlp* m, float* host) {
    if (!m || !host) return TSM_ERR_INVALID_VALUE;
    return cudaMemcpy(host, m->params, sizeof(float) * m->P, cudaMemcpyDeviceToHost) == cudaSuccess
               ? TSM_OK
               : TSM_ERR_LAUNCH;
}

tsm_status tsm_mlp_get_grads(const tsm_mlp* m, float* host) {
    if (!m || !host) return TSM_ERR_INVALID_VALUE;
    return cudaMemcpy(host, m->grads, sizeof(float) * m->P, cudaMemcpyDeviceToHost) == cudaSuccess
               ? TSM_OK
               : TSM_ERR_LAUNCH;
}

tsm_status tsm_mlp_forward(tsm_mlp* m, const float* X, int n, float* y, tsm_stream_t stream) {
    if (!m || !X || !y || n < 1 || n > m->max_batch) return TSM_ERR_INVALID_VALUE;
    const size_t smem = offsetof(mlp::Smem, W2T);
    if (cudaFuncSetAttribute(mlp::k_mlp<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
        cudaSuccess)
        return TSM_ERR_LAUNCH;
    const int tiles = (n - 1) / mlp::TS + 1;
    mlp::k_mlp<false><<<std::min(tiles, m->grid_max), mlp::kThreads, smem, (cudaStream_t)stream>>>(
        m->params, m->D, m->H, X, nullptr, n, y, nullptr, nullptr);
    return cudaGetLastError() == cudaSuccess ? TSM_OK : TSM_ERR_LAUNCH;
}

tsm_status tsm_mlp_backward(tsm_mlp* m, const float* X, const float* t, int n, float* loss,
                            tsm_stream_t stream) {
    if (!m || !X || !t || !loss || n < 1 || n > m->max_batch) return TSM_ERR_INVALID_VALUE;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t smem = sizeof(mlp::Smem);
    if (cudaFuncSetAttribute(mlp::k_mlp<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return TSM_ERR_LAUNCH;
    const int grid = std::min((n - 1) / mlp::TS + 1, m->grid_max);
    mlp::k_mlp<true><<<grid, mlp::kThreads, smem, s>>>(m->params, m->D, m->H, X, t, n, nullptr, m->parts, m->lparts);
    mlp::k_mlp_sum<<<(m->P + 31) / 32 + 1, 32 * mlp::kSlices, 0, s>>>(m->parts, m->lparts, grid, m->P, n, m->grads,
                                                                      loss);
    return cudaGetLastError() == cudaSuccess ? TSM_OK : TSM_ERR_LAUNCH;
}

tsm_status tsm_mlp_adam(tsm_mlp* m, float lr, float beta1, float beta2, float eps, tsm_stream_t stream) {
    if (!m || !(lr > 0.0f) || !(beta1 >= 0.0f && beta1 < 1.0f) || !(beta2 >= 0.0f && beta2 < 1.0f) ||
        !(eps > 0.0f))
        return TSM_ERR_INVALID_VALUE;
    m->step += 1;
    const float c1 = 1.0f - powf(beta1, (float)m->step);
    const float c2 = 1.0f - powf(beta2, (float)m->step);
    mlp::k_adam<<<(m->P + 127) / 128, 128, 0, (cudaStream_t)stream>>>(m->params, m->grads, m->m, m->v, m->P, lr,
                                                                      beta1, beta2, eps, c1, c2);
    return cudaGetLastError() == cudaSuccess ? TSM_OK : TSM_ERR_LAUNCH;
}

}  // extern "C"
