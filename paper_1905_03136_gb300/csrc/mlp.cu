// The cost model's network: 3-layer tanh perceptron, FP32, with hand-written
// forward, backward and Adam kernels (see tsm_mlp.h for the maths and the
// parameter layout).
//
// A call is a few hundred MFLOP at most (6126 samples, 17-64-64-1: 0.18
// GFLOP, 2.6 us at the FP32 rate), so what bounds it is latency: how many
// threads share the work, and how long the serial chains are.  Forward and
// gradient run as one kernel over tiles of 16 samples whose weights and
// activations stay in shared memory; each thread owns a small register tile
// of every layer product (2 samples x 4 units, 8 x 4 weights), the output unit
// and all that follows from it alone stay in the threads of their sample, and
// the CTA adds up its samples' share of the gradient in registers.  A second
// kernel, started early, sums the CTA shares.  Every order is fixed, so
// results repeat bit for bit.  Tiles of 32 samples and CTAs of 256 threads
// left 112 of 152 SMs with one CTA and 40 with two (27 us for the kernel).
// Measured (6126 samples, D = 17, H = 64, loss and gradient with its copy to
// the host): 1415 us with one thread per sample and one per parameter over
// all samples (a chain of 6126 dependent FMAs), 43 to 49 us now.
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>
#include <utility>
#include <vector>

#include "fp64_common.cuh"
#include "tsm_internal.h"
#include "tsm_mlp.h"

struct tsm_mlp {
    int D, H, max_batch, P;
    float* params;  // device
    float* grads;
    float* m;
    float* v;
    float* parts;   // grid_max x stride: the CTAs' shares of the gradient
    double* lparts; // grid_max: their shares of the squared error
    int grid_max;   // CTAs the shares are sized for
    int stride;     // P rounded up to a multiple of four
    int64_t step;
    mutable std::mutex mu;
    mutable std::vector<std::pair<cudaStream_t, cudaEvent_t>> used;  // last work on each other stream than the legacy one
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

constexpr int kThreads = 128;
constexpr int TS = 16;              // samples per tile
constexpr int TY = 8;               // thread rows: samples ty and ty + 8, weight rows 8 ty ..
constexpr int HMAX = TSM_MLP_MAX_HIDDEN, DMAX = TSM_MLP_MAX_IN;
constexpr int HS = HMAX + 4;        // row strides in floats: 16-byte aligned, and eight
constexpr int DS = DMAX + 4;        // consecutive rows fall into different banks
constexpr int kCtasPerSm = 4;       // resident CTAs of either kernel (49 KB of shared memory each)
static_assert(HMAX == 64 && DMAX == 32 && TS == 2 * TY && kThreads == 16 * TY, "the thread tiles cover these");

// Shared memory of one CTA.  Rows and columns past H, D and the tile's
// samples hold zeros.
struct Smem {
    float W1[HMAX][DS], W2[HMAX][HS];
    float b1[HMAX], b2[HMAX], w3[HMAX];
    float x[TS][DS], h1[TS][HS];
    // gradient only
    float d1[TS][HS], d2[TS][HS];
    float red[3][TY][HMAX];  // b1, b2, w3: the thread rows' sums
    double lsum[TY];
    float dsum[TY];
};

// out[a][b] += sum over k < n4 (a multiple of 4) of X[s + 8a][k] W[u + 16b][k],
// k ascending: two LDS.128 of samples (broadcast) and four of weights feed
// 32 FMAs.
template <int XS, int WS>
__device__ __forceinline__ void layer(const float (*X)[XS], const float (*W)[WS], int n4, int s, int u,
                                      float (&out)[2][4]) {
#pragma unroll 2
    for (int k = 0; k < n4; k += 4) {
        float4 xv[2], wv[4];
#pragma unroll
        for (int a = 0; a < 2; ++a) xv[a] = *reinterpret_cast<const float4*>(&X[s + TY * a][k]);
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
// gradient (parts + blockIdx.x * stride) and of the squared error.  CTA b
// takes tiles b, b + gridDim.x, ...
template <bool GRAD>
__global__ void __launch_bounds__(kThreads, kCtasPerSm) k_mlp(const float* __restrict__ p, int D, int H,
                                                              const float* __restrict__ X,
                                                              const float* __restrict__ target, int n,
                                                              float* __restrict__ y, float* __restrict__ parts,
                                                              int stride, double* __restrict__ lparts) {
    extern __shared__ __align__(16) unsigned char raw[];
    Smem& S = *reinterpret_cast<Smem*>(raw);
    if (GRAD) pdl_trigger();
    const Off o = offsets(D, H);
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int H4 = (H + 3) & ~3, D4 = (D + 3) & ~3;
    // the first tile's samples are on their way while the weights are staged
    float xr[TS * DMAX / kThreads], tr[2] = {0.0f, 0.0f};
    auto fetch = [&](int tile) {
        const int i0 = tile * TS;
#pragma unroll
        for (int c = 0; c < TS * DMAX / kThreads; ++c) {
            const int i = tid + c * kThreads, s = i / DMAX, k = i - s * DMAX;
            xr[c] = i0 + s < n && k < D ? X[(int64_t)(i0 + s) * D + k] : 0.0f;
        }
#pragma unroll
        for (int a = 0; a < 2; ++a)
            if (GRAD) tr[a] = i0 + ty + TY * a < n ? target[i0 + ty + TY * a] : 0.0f;
    };
    const int tiles = (n + TS - 1) / TS;
    fetch(blockIdx.x);
#pragma unroll
    for (int c = 0; c < HMAX * DMAX / kThreads; ++c) {
        const int i = tid + c * kThreads, j = i / DMAX, k = i - j * DMAX;
        S.W1[j][k] = j < H && k < D ? p[o.W1 + j * D + k] : 0.0f;
    }
#pragma unroll
    for (int c = 0; c < HMAX * HMAX / kThreads; ++c) {
        const int i = tid + c * kThreads, j = i / HMAX, k = i - j * HMAX;
        S.W2[j][k] = j < H && k < H ? p[o.W2 + j * H + k] : 0.0f;
    }
    if (tid < HMAX) {
        S.b1[tid] = tid < H ? p[o.b1 + tid] : 0.0f;
        S.b2[tid] = tid < H ? p[o.b2 + tid] : 0.0f;
        S.w3[tid] = tid < H ? p[o.w3 + tid] : 0.0f;
    }
    const float b3 = p[o.b3];
    // gradient sums of this thread: W2[8ty + r][4tx + c], W1[8ty + r][tx + 16c],
    // and its samples' part of b1[4tx + c], b2 and w3[tx + 16b], b3
    float gW2[8][4] = {}, gW1[8][2] = {}, gb1[4] = {}, gb2[4] = {}, gw3[4] = {}, gb3 = 0.0f;
    double lsum = 0.0;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int i0 = tile * TS;
        __syncthreads();  // the previous tile is done with
#pragma unroll
        for (int c = 0; c < TS * DMAX / kThreads; ++c) {
            const int i = tid + c * kThreads, s = i / DMAX, k = i - s * DMAX;
            S.x[s][k] = xr[c];
        }
        const float t0[2] = {tr[0], tr[1]};
        if (tile + (int)gridDim.x < tiles) fetch(tile + gridDim.x);
        __syncthreads();  // (first tile: and the weights are staged)
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
            for (int b = 0; b < 4; ++b) S.h1[ty + TY * a][tx + 16 * b] = tx + 16 * b < H ? tanhf(v[a][b]) : 0.0f;
        __syncthreads();
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) v[a][b] = S.b2[tx + 16 * b];
        layer(S.h1, S.W2, H4, ty, tx, v);
        // the output unit: this thread's four units, then the 16 threads of
        // the sample in a fixed tree
        float w3[4], yv[2] = {0.0f, 0.0f};
#pragma unroll
        for (int b = 0; b < 4; ++b) w3[b] = S.w3[tx + 16 * b];
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                v[a][b] = tx + 16 * b < H ? tanhf(v[a][b]) : 0.0f;
                yv[a] = fmaf(w3[b], v[a][b], yv[a]);
            }
#pragma unroll
        for (int h = 8; h >= 1; h >>= 1)
#pragma unroll
            for (int a = 0; a < 2; ++a) yv[a] += __shfl_xor_sync(0xffffffffu, yv[a], h);
        if constexpr (!GRAD) {
#pragma unroll
            for (int a = 0; a < 2; ++a)
                if (tx == 0 && i0 + ty + TY * a < n) y[i0 + ty + TY * a] = b3 + yv[a];
            continue;
        }
        // dL/d(pre-activation of layer 2), and the sums over the samples of
        // what multiplies b2, w3 and b3
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const int s = ty + TY * a;
            const float e = i0 + s < n ? b3 + yv[a] - t0[a] : 0.0f;
            const float dy = 2.0f * e / (float)n;
            lsum += (double)(e * e);
            gb3 += dy;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const float d = tx + 16 * b < H ? dy * w3[b] * (1.0f - v[a][b] * v[a][b]) : 0.0f;
                S.d2[s][tx + 16 * b] = d;
                gb2[b] += d;
                gw3[b] = fmaf(dy, v[a][b], gw3[b]);
                v[a][b] = 0.0f;
            }
        }
        __syncthreads();
        // ... and of layer 1, units 4tx + c: sum over j of W2[j][4tx + c] d2[j],
        // j ascending
#pragma unroll 2
        for (int j = 0; j < H4; j += 4) {
            float4 dv[2], wv[4];
#pragma unroll
            for (int a = 0; a < 2; ++a) dv[a] = *reinterpret_cast<const float4*>(&S.d2[ty + TY * a][j]);
#pragma unroll
            for (int i = 0; i < 4; ++i) wv[i] = *reinterpret_cast<const float4*>(&S.W2[j + i][4 * tx]);
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                const float dd[4] = {dv[a].x, dv[a].y, dv[a].z, dv[a].w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    v[a][0] = fmaf(wv[i].x, dd[i], v[a][0]);
                    v[a][1] = fmaf(wv[i].y, dd[i], v[a][1]);
                    v[a][2] = fmaf(wv[i].z, dd[i], v[a][2]);
                    v[a][3] = fmaf(wv[i].w, dd[i], v[a][3]);
                }
            }
        }
#pragma unroll
        for (int a = 0; a < 2; ++a) {
            const float4 h = *reinterpret_cast<const float4*>(&S.h1[ty + TY * a][4 * tx]);
            const float4 d = make_float4(v[a][0] * (1.0f - h.x * h.x), v[a][1] * (1.0f - h.y * h.y),
                                         v[a][2] * (1.0f - h.z * h.z), v[a][3] * (1.0f - h.w * h.w));
            *reinterpret_cast<float4*>(&S.d1[ty + TY * a][4 * tx]) = d;
            gb1[0] += d.x;
            gb1[1] += d.y;
            gb1[2] += d.z;
            gb1[3] += d.w;
        }
        __syncthreads();
        // the tile's samples added to this thread's weight entries (those past
        // n have d1 = d2 = 0)
#pragma unroll 2
        for (int s = 0; s < TS; ++s) {
            const float4 h = *reinterpret_cast<const float4*>(&S.h1[s][4 * tx]);
            const float x0 = S.x[s][tx], x1 = S.x[s][tx + 16];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const float4 d = *reinterpret_cast<const float4*>(&S.d2[s][8 * ty + 4 * q]);
                const float4 e = *reinterpret_cast<const float4*>(&S.d1[s][8 * ty + 4 * q]);
                const float dv[4] = {d.x, d.y, d.z, d.w}, ev[4] = {e.x, e.y, e.z, e.w};
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    gW2[4 * q + r][0] = fmaf(dv[r], h.x, gW2[4 * q + r][0]);
                    gW2[4 * q + r][1] = fmaf(dv[r], h.y, gW2[4 * q + r][1]);
                    gW2[4 * q + r][2] = fmaf(dv[r], h.z, gW2[4 * q + r][2]);
                    gW2[4 * q + r][3] = fmaf(dv[r], h.w, gW2[4 * q + r][3]);
                    gW1[4 * q + r][0] = fmaf(ev[r], x0, gW1[4 * q + r][0]);
                    gW1[4 * q + r][1] = fmaf(ev[r], x1, gW1[4 * q + r][1]);
                }
            }
        }
    }
    if (!GRAD) return;
    float* g = parts + (int64_t)blockIdx.x * stride;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const int j = 8 * ty + r;
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (j < H && 4 * tx + c < H) g[o.W2 + j * H + 4 * tx + c] = gW2[r][c];
#pragma unroll
        for (int c = 0; c < 2; ++c)
            if (j < H && tx + 16 * c < D) g[o.W1 + j * D + tx + 16 * c] = gW1[r][c];
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        S.red[0][ty][4 * tx + c] = gb1[c];
        S.red[1][ty][tx + 16 * c] = gb2[c];
        S.red[2][ty][tx + 16 * c] = gw3[c];
    }
    if (tx == 0) {
        S.dsum[ty] = gb3;
        S.lsum[ty] = lsum;
    }
    __syncthreads();
    for (int i = tid; i < 3 * HMAX; i += kThreads) {
        const int q = i / HMAX, j = i - q * HMAX;
        float s = 0.0f;
#pragma unroll
        for (int r = 0; r < TY; ++r) s += S.red[q][r][j];
        if (j < H) g[(q == 0 ? o.b1 : (q == 1 ? o.b2 : o.w3)) + j] = s;
    }
    if (tid == kThreads - 1) {
        float s = 0.0f;
        double l = 0.0;
#pragma unroll
        for (int r = 0; r < TY; ++r) {
            s += S.dsum[r];
            l += S.lsum[r];
        }
        g[o.b3] = s;
        lparts[blockIdx.x] = l;
    }
}

// Gradient and loss from the CTAs' shares (rows of `stride` floats, a multiple
// of four).  A thread takes four parameters of shares r, r + 32, ... in order,
// and the 32 sums are combined by a fixed-pairing tree; the last CTA does the
// same for the loss, in double.  Bound by the latency of the shares' reads
// from L2: few of them in a thread's chain, all of them wide.
constexpr int kSlices = 32, kQuads = 8;
__global__ void __launch_bounds__(kSlices * kQuads) k_mlp_sum(const float* __restrict__ parts, int stride,
                                                              const double* __restrict__ lparts, int G, int P, int n,
                                                              float* __restrict__ g, float* __restrict__ loss) {
    __shared__ float4 red[kSlices][kQuads];
    const int t = threadIdx.x, c = t % kQuads, r = t / kQuads;
    pdl_wait();  // starts while k_mlp runs
    if (blockIdx.x == gridDim.x - 1) {
        double* dr = reinterpret_cast<double*>(&red[0][0]);
        double s = 0.0;
        for (int b = t; b < G; b += kSlices * kQuads) s += lparts[b];
        dr[t] = s;
        __syncthreads();
        for (int h = kSlices * kQuads / 2; h >= 1; h >>= 1) {
            if (t < h) dr[t] += dr[t + h];
            __syncthreads();
        }
        if (t == 0) *loss = (float)(dr[0] / n);
        return;
    }
    const int q = (blockIdx.x * kQuads + c) * 4;
    float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (q < P) {
#pragma unroll 8
        for (int b = r; b < G; b += kSlices) {
            const float4 x = *reinterpret_cast<const float4*>(parts + (int64_t)b * stride + q);
            s.x += x.x;
            s.y += x.y;
            s.z += x.z;
            s.w += x.w;
        }
    }
    red[r][c] = s;
    __syncthreads();
    for (int h = kSlices / 2; h >= 1; h >>= 1) {
        if (r < h) {
            float4 a = red[r][c];
            const float4 b = red[r + h][c];
            a.x += b.x;
            a.y += b.y;
            a.z += b.z;
            a.w += b.w;
            red[r][c] = a;
        }
        __syncthreads();
    }
    if (t < 4 * kQuads) {
        const int w = blockIdx.x * 4 * kQuads + t;
        if (w < P) g[w] = reinterpret_cast<const float*>(&red[0][0])[t];
    }
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

// The host copies run on the legacy stream, which non-blocking streams do not
// wait for, nor it for them.  note_use records where a stream's last work on
// the model ends; the next copy has the legacy stream wait for all of them
// and forgets them.  (Work being captured runs when its graph does: the
// caller orders that.)
cudaError_t note_use(tsm_mlp* m, cudaStream_t s) try {
    if (s == nullptr || s == cudaStreamLegacy) return cudaSuccess;
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(s, &st);
    if (e != cudaSuccess || st != cudaStreamCaptureStatusNone) return e;
    std::lock_guard<std::mutex> lock(m->mu);
    for (const auto& u : m->used)
        if (u.first == s) return cudaEventRecord(u.second, s);
    m->used.reserve(m->used.size() + 1);
    cudaEvent_t ev = nullptr;
    if ((e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming)) != cudaSuccess) return e;
    m->used.emplace_back(s, ev);
    return cudaEventRecord(ev, s);
} catch (...) {
    return cudaErrorMemoryAllocation;
}
cudaError_t join_uses(const tsm_mlp* m) {
    std::lock_guard<std::mutex> lock(m->mu);
    for (const auto& u : m->used) {
        const cudaError_t e = cudaStreamWaitEvent(nullptr, u.second, 0);
        if (e != cudaSuccess) return e;
    }
    for (const auto& u : m->used) cudaEventDestroy(u.second);
    m->used.clear();
    return cudaSuccess;
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
    tsm_mlp* m = new (std::nothrow) tsm_mlp();
    if (!m) return TSM_ERR_ALLOC;
    const mlp::Off o = mlp::offsets(in_dim, hidden);
    m->D = in_dim;
    m->H = hidden;
    m->max_batch = max_batch;
    m->P = o.P;
    m->stride = (o.P + 3) & ~3;
    const size_t pb = sizeof(float) * o.P;
    // one share per CTA: a resident wave, or fewer tiles than that
    const int sms = device_info().sm_count;
    m->grid_max = std::max(1, std::min((max_batch - 1) / mlp::TS + 1, mlp::kCtasPerSm * sms));
    bool ok = cudaMalloc(&m->params, pb) == cudaSuccess && cudaMalloc(&m->grads, pb) == cudaSuccess &&
              cudaMalloc(&m->m, pb) == cudaSuccess && cudaMalloc(&m->v, pb) == cudaSuccess &&
              cudaMalloc(&m->parts, sizeof(float) * m->stride * m->grid_max) == cudaSuccess &&
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
    // in place before this returns, whatever stream the model is used on
    cudaStream_t cs = nullptr;
    ok = setup_stream(&cs) == cudaSuccess &&
         cudaMemcpyAsync(m->params, h.data(), pb, cudaMemcpyHostToDevice, cs) == cudaSuccess &&
         cudaMemsetAsync(m->grads, 0, pb, cs) == cudaSuccess && cudaMemsetAsync(m->m, 0, pb, cs) == cudaSuccess &&
         cudaMemsetAsync(m->v, 0, pb, cs) == cudaSuccess;
    if (cs) ok = cudaStreamSynchronize(cs) == cudaSuccess && ok;
    if (!ok) {
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
    for (const auto& u : m->used) cudaEventDestroy(u.second);
    delete m;
}

int tsm_mlp_param_count(const tsm_mlp* m) { return m ? m->P : -1; }

tsm_status tsm_mlp_set_params(tsm_mlp* m, const float* host) {
    if (!m || !host) return TSM_ERR_INVALID_VALUE;
    if (mlp::join_uses(m) != cudaSuccess) return TSM_ERR_LAUNCH;
    if (cudaMemcpy(m->params, host, sizeof(float) * m->P, cudaMemcpyHostToDevice) != cudaSuccess)
        return TSM_ERR_LAUNCH;
    // a new parameter vector restarts the optimiser
    if (cudaMemset(m->m, 0, sizeof(float) * m->P) != cudaSuccess ||
        cudaMemset(m->v, 0, sizeof(float) * m->P) != cudaSuccess || cudaStreamSynchronize(nullptr) != cudaSuccess)
        return TSM_ERR_LAUNCH;
    m->step = 0;
    return TSM_OK;
}

tsm_status tsm_mlp_get_params(const tsm_mlp* m, float* host) {
    if (!m || !host) return TSM_ERR_INVALID_VALUE;
    if (mlp::join_uses(m) != cudaSuccess) return TSM_ERR_LAUNCH;
    return cudaMemcpy(host, m->params, sizeof(float) * m->P, cudaMemcpyDeviceToHost) == cudaSuccess
               ? TSM_OK
               : TSM_ERR_LAUNCH;
}

tsm_status tsm_mlp_get_grads(const tsm_mlp* m, float* host) {
    if (!m || !host) return TSM_ERR_INVALID_VALUE;
    if (mlp::join_uses(m) != cudaSuccess) return TSM_ERR_LAUNCH;
    return cudaMemcpy(host, m->grads, sizeof(float) * m->P, cudaMemcpyDeviceToHost) == cudaSuccess
               ? TSM_OK
               : TSM_ERR_LAUNCH;
}

tsm_status tsm_mlp_forward(tsm_mlp* m, const float* X, int n, float* y, tsm_stream_t stream) {
    if (!m || !X || !y || n < 1 || n > m->max_batch) return TSM_ERR_INVALID_VALUE;
    const size_t smem = offsetof(mlp::Smem, d1);
    if (cudaFuncSetAttribute(mlp::k_mlp<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
        cudaSuccess)
        return TSM_ERR_LAUNCH;
    const int tiles = (n - 1) / mlp::TS + 1;
    mlp::k_mlp<false><<<std::min(tiles, m->grid_max), mlp::kThreads, smem, (cudaStream_t)stream>>>(
        m->params, m->D, m->H, X, nullptr, n, y, nullptr, 0, nullptr);
    if (cudaGetLastError() != cudaSuccess) return TSM_ERR_LAUNCH;
    return mlp::note_use(m, (cudaStream_t)stream) == cudaSuccess ? TSM_OK : TSM_ERR_LAUNCH;
}

tsm_status tsm_mlp_backward(tsm_mlp* m, const float* X, const float* t, int n, float* loss,
                            tsm_stream_t stream) {
    if (!m || !X || !t || !loss || n < 1 || n > m->max_batch) return TSM_ERR_INVALID_VALUE;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t smem = sizeof(mlp::Smem);
    if (cudaFuncSetAttribute(mlp::k_mlp<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return TSM_ERR_LAUNCH;
    const int grid = std::min((n - 1) / mlp::TS + 1, m->grid_max);
    mlp::k_mlp<true><<<grid, mlp::kThreads, smem, s>>>(m->params, m->D, m->H, X, t, n, nullptr, m->parts, m->stride,
                                                       m->lparts);
    if (cudaGetLastError() != cudaSuccess) return TSM_ERR_LAUNCH;
    const int quads = (m->P + 4 * mlp::kQuads - 1) / (4 * mlp::kQuads);
    if (launch_early(pdl_enabled(), mlp::k_mlp_sum, quads + 1, mlp::kSlices * mlp::kQuads, 0, s, m->parts, m->stride,
                     m->lparts, grid, m->P, n, m->grads, loss) != cudaSuccess)
        return TSM_ERR_LAUNCH;
    return mlp::note_use(m, s) == cudaSuccess ? TSM_OK : TSM_ERR_LAUNCH;
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
    if (cudaGetLastError() != cudaSuccess) return TSM_ERR_LAUNCH;
    return mlp::note_use(m, (cudaStream_t)stream) == cudaSuccess ? TSM_OK : TSM_ERR_LAUNCH;
}

}  // extern "C"
