// Learned probe depth: a small MLP predicts, per query, the depth p that
// reproduces the top-k of a large fixed depth.  Not in the paper, where the
// probe depth is one fixed number per subindex (Algorithm 2); the fixed-depth
// method stays as the fallback and as the source of the training labels.
//
//   features   4 per curve: octave encodings of the key gaps to the list
//              neighbours of the query key, and of the min / mean distance of
//              the 8 list entries around it (exact, integer-derived values)
//   labels     minimal p in [0, p_max] whose top-k equals the top-k at p_max:
//              the depth at which the last of those neighbours enters a window
//   model      x^ = (x - mu) * isd;  h1 = relu(x^ W1 + b1);
//              h2 = relu(h1 W2 + b2);  y = h2 . W3 + b3   (y ~ log2 p)
//   training   two FP32 kernels per step: the layers forward and back for 32
//              samples per block, then every weight's gradient and Adam update
//   inference  BF16 inputs and weights, FP32 accumulation, fused with the
//              feature computation: one, two or four queries per warp
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "hc_index.h"
#include "hc_trace.h"
#include "hc_query_dev.cuh"

using namespace hc;

// ---------------------------------------------------------------- model
struct hc_mlp {
    uint32_t in = 0, h1 = 0, h2 = 0, max_batch = 0;
    uint32_t nparam = 0;          // trained parameters
    float* params = nullptr;      // device: W1 b1 W2 b2 W3 b3 | mu isd
    float* grads = nullptr;
    float* adam_m = nullptr;
    float* adam_v = nullptr;
    __nv_bfloat16* wbf = nullptr; // device: W1 W2 W3 in bf16 (inference)
    float* work = nullptr;        // device: a batch's activations (Work)
    float* loss = nullptr;        // device scalar
    uint64_t steps = 0;
    bool bf_stale = true;
};

namespace {

struct Layout {
    uint32_t W1, b1, W2, b2, W3, b3, mu, isd, total_trained, total;
};

Layout layout_of(uint32_t in, uint32_t h1, uint32_t h2) {
    Layout L;
    L.W1 = 0;
    L.b1 = L.W1 + in * h1;
    L.W2 = L.b1 + h1;
    L.b2 = L.W2 + h1 * h2;
    L.W3 = L.b2 + h2;
    L.b3 = L.W3 + h2;
    L.total_trained = L.b3 + 1;
    L.mu = L.total_trained;
    L.isd = L.mu + in;
    L.total = L.isd + in;
    return L;
}

// What one training step's forward and backward pass leaves in hc_mlp::work for
// the weight gradients: a row per unit, a column per sample (pitch: max_batch
// rounded up to 64), so that a gradient's sum over the samples reads rows.
// loss: one partial sum per kTile samples.
constexpr uint32_t kTile = 32;   // samples per block of the layer pass

struct Work {
    uint32_t pitch = 0;
    float *xn = nullptr, *a1 = nullptr, *a2 = nullptr, *dy = nullptr, *d2 = nullptr,
          *d1 = nullptr, *loss = nullptr;
};

uint32_t work_pitch(uint32_t max_batch) { return (max_batch + 63) / 64 * 64; }

Work work_of(const hc_mlp* M) {
    Work w;
    const size_t B = w.pitch = work_pitch(M->max_batch);
    w.xn = M->work;
    w.a1 = w.xn + B * M->in;
    w.a2 = w.a1 + B * M->h1;
    w.dy = w.a2 + B * M->h2;
    w.d2 = w.dy + B;
    w.d1 = w.d2 + B * M->h2;
    w.loss = w.d1 + B * M->h1;
    return w;
}

size_t work_floats(uint32_t in, uint32_t h1, uint32_t h2, uint32_t max_batch) {
    const size_t B = work_pitch(max_batch);
    return B * (in + 2 * h1 + 2 * h2 + 1) + B / kTile;
}

constexpr uint32_t kMaxDim = 64;

// Shared memory of the layer pass: the weights (units past a layer's width are
// zero) and the tile's activations, rows of kPitch floats: 16-byte aligned, and
// eight rows apart by 4 banks each, so a 16-byte column of eight rows is read
// without a conflict.
constexpr uint32_t kPitch = kMaxDim + 4;
struct LayerSmem {
    float w1[kMaxDim][kPitch], w2[kMaxDim][kPitch];
    float w3[kMaxDim], b1[kMaxDim], b2[kMaxDim];
    float x[kTile][kPitch], a1[kTile][kPitch], a2[kTile][kPitch], d2[kTile][kPitch];
    float dy[kTile];
};

// acc[s][c] = sum over k < K (rounded up to 4; the padding is zero) of
// in[2 ty + s][k] w[k][4 tx + c], k ascending
__device__ __forceinline__ void layer_tile(const float (*in)[kPitch], const float (*w)[kPitch],
                                           uint32_t K, uint32_t tx, uint32_t ty,
                                           float (&acc)[2][4]) {
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[s][c] = 0.f;
    for (uint32_t k = 0; k < K; k += 4) {
        float x[2][4], v[4][4];
#pragma unroll
        for (int s = 0; s < 2; ++s)
            *reinterpret_cast<float4*>(x[s]) =
                *reinterpret_cast<const float4*>(&in[2 * ty + s][k]);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            *reinterpret_cast<float4*>(v[j]) = *reinterpret_cast<const float4*>(&w[k + j][4 * tx]);
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[s][c] = fmaf(x[s][j], v[j][c], acc[s][c]);
    }
}

struct LayerArgs {
    Layout L;
    const float* P;            // parameters, then mu and isd
    uint32_t in, h1, h2, n;    // n samples, kTile per block
    const float* x;            // rows of `in` features
    const float* t;            // targets (training)
    const uint32_t* perm;      // sample i is row perm[i] of x and t, or i when null
    float* y;                  // outputs (inference), or null: training
    Work w;
};

// The layers for kTile samples per block: forward, and for training the
// gradients of the activations back to the first layer.  Weights and
// activations stay in shared memory (one read of the weights per block); a
// thread computes two samples by four units per layer, every sum in order of
// its index, and a training step's activations leave transposed.  Bound by the
// latency of the five dependent layers (40 steps of shared-memory loads and
// FMAs, two warps per scheduler) and the shared-memory wavefronts (8,000 cycles):
// 10.6 us for 4096 samples on 128 blocks.
__global__ void __launch_bounds__(256) layers_kernel(LayerArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    LayerSmem& sm = *reinterpret_cast<LayerSmem*>(smem_raw);
    const uint32_t tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
    const uint32_t m0 = blockIdx.x * kTile;
    const float *mu = a.P + a.L.mu, *isd = a.P + a.L.isd;
    // all global loads of the staging in flight at once
    constexpr uint32_t kW = kMaxDim * kMaxDim / 256, kX = kTile * kMaxDim / 256;
    const uint32_t col = tid % kMaxDim, row0 = tid / kMaxDim;   // rows row0 + 4 u
    float xv[kX], w1v[kW], w2v[kW];
#pragma unroll
    for (uint32_t u = 0; u < kX; ++u) {
        const uint32_t i = m0 + row0 + 4 * u;
        xv[u] = i < a.n && col < a.in ? a.x[(size_t)(a.perm ? a.perm[i] : i) * a.in + col] : 0.f;
    }
    float target = 0.f;
    if (!a.y && tid < kTile && m0 + tid < a.n) target = a.t[a.perm ? a.perm[m0 + tid] : m0 + tid];
    const float b3 = a.P[a.L.b3];
#pragma unroll
    for (uint32_t u = 0; u < kW; ++u) {
        const uint32_t r = row0 + 4 * u;
        w1v[u] = r < a.in && col < a.h1 ? a.P[a.L.W1 + r * a.h1 + col] : 0.f;
        w2v[u] = r < a.h1 && col < a.h2 ? a.P[a.L.W2 + r * a.h2 + col] : 0.f;
    }
    const float mu_c = col < a.in ? mu[col] : 0.f, isd_c = col < a.in ? isd[col] : 0.f;
#pragma unroll
    for (uint32_t u = 0; u < kW; ++u) {
        sm.w1[row0 + 4 * u][col] = w1v[u];
        sm.w2[row0 + 4 * u][col] = w2v[u];
    }
    if (tid < kMaxDim) {
        sm.w3[tid] = tid < a.h2 ? a.P[a.L.W3 + tid] : 0.f;
        sm.b1[tid] = tid < a.h1 ? a.P[a.L.b1 + tid] : 0.f;
        sm.b2[tid] = tid < a.h2 ? a.P[a.L.b2 + tid] : 0.f;
    }
#pragma unroll
    for (uint32_t u = 0; u < kX; ++u)
        sm.x[row0 + 4 * u][col] =
            m0 + row0 + 4 * u < a.n && col < a.in ? (xv[u] - mu_c) * isd_c : 0.f;
    __syncthreads();
    float acc[2][4];
    layer_tile(sm.x, sm.w1, a.in, tx, ty, acc);
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int c = 0; c < 4; ++c)
            sm.a1[2 * ty + s][4 * tx + c] = fmaxf(acc[s][c] + sm.b1[4 * tx + c], 0.f);
    __syncthreads();
    layer_tile(sm.a1, sm.w2, a.h1, tx, ty, acc);
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int c = 0; c < 4; ++c)
            sm.a2[2 * ty + s][4 * tx + c] = fmaxf(acc[s][c] + sm.b2[4 * tx + c], 0.f);
    __syncthreads();
    if (tid < kTile) {
        const bool real = m0 + tid < a.n;
        float y = 0.f;
#pragma unroll 4
        for (uint32_t j = 0; j < a.h2; j += 4) {   // past the layer: zeros
            const float4 h = *reinterpret_cast<const float4*>(&sm.a2[tid][j]);
            const float4 w = *reinterpret_cast<const float4*>(&sm.w3[j]);
            y = fmaf(h.x, w.x, y);
            y = fmaf(h.y, w.y, y);
            y = fmaf(h.z, w.z, y);
            y = fmaf(h.w, w.w, y);
        }
        y += b3;
        if (a.y) {
            if (real) a.y[m0 + tid] = y;
        } else {
            const float e = real ? y - target : 0.f;
            const float dy = 2.f * e / (float)a.n;
            float l = e * e / (float)a.n;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
            if (tid == 0) a.w.loss[blockIdx.x] = l;
            sm.dy[tid] = dy;
            a.w.dy[m0 + tid] = dy;
        }
    }
    if (a.y) return;
    __syncthreads();
    // d2 = (dy W3^T) * [a2 > 0]
    for (uint32_t i = tid; i < kTile * kMaxDim; i += 256) {
        const uint32_t s = i / kMaxDim, c = i % kMaxDim;
        sm.d2[s][c] = sm.a2[s][c] > 0.f ? fmaf(sm.dy[s], sm.w3[c], 0.f) : 0.f;
    }
    __syncthreads();
    // d1 = (d2 W2^T) * [a1 > 0]: unit tx + 16 c of samples 2 ty, 2 ty + 1
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[s][c] = 0.f;
    for (uint32_t k = 0; k < a.h2; k += 4) {
        float g[2][4], v[4][4];
#pragma unroll
        for (int s = 0; s < 2; ++s)
            *reinterpret_cast<float4*>(g[s]) =
                *reinterpret_cast<const float4*>(&sm.d2[2 * ty + s][k]);
#pragma unroll
        for (int c = 0; c < 4; ++c)
            *reinterpret_cast<float4*>(v[c]) =
                *reinterpret_cast<const float4*>(&sm.w2[tx + 16 * c][k]);
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int s = 0; s < 2; ++s)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[s][c] = fmaf(g[s][j], v[c][j], acc[s][c]);
    }
    __syncthreads();   // sm.w1 makes room for d1
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int c = 0; c < 4; ++c)
            sm.w1[2 * ty + s][tx + 16 * c] =
                sm.a1[2 * ty + s][tx + 16 * c] > 0.f ? acc[s][c] : 0.f;
    __syncthreads();
    // samples past the batch leave zeros, which add nothing to a gradient
    const uint32_t lane = tid % 32, warp = tid / 32;
    const bool real = m0 + lane < a.n;
    auto put = [&](float* rows, uint32_t units, const float (*src)[kPitch]) {
        for (uint32_t u = warp; u < units; u += 8)
            rows[(size_t)u * a.w.pitch + m0 + lane] = real ? src[lane][u] : 0.f;
    };
    put(a.w.xn, a.in, sm.x);
    put(a.w.a1, a.h1, sm.a1);
    put(a.w.a2, a.h2, sm.a2);
    put(a.w.d2, a.h2, sm.d2);
    put(a.w.d1, a.h1, sm.w1);
}

// Adam (beta 0.9 / 0.999, eps 1e-8) with the bias corrections of the step
struct Adam {
    float lr, beta1, beta2, eps, corr1, corr2;
};

struct GradArgs {
    Layout L;
    uint32_t in, h1, h2, n;
    Work w;
    float *P, *G, *m, *v;
    bool update;   // also one Adam step
    Adam adam;
};

__device__ __forceinline__ void take_gradient(const GradArgs& a, uint32_t i, float gi) {
    a.G[i] = gi;
    if (!a.update) return;
    const float mi = __fmaf_rn(1.f - a.adam.beta1, gi, __fmul_rn(a.adam.beta1, a.m[i]));
    const float vi =
        __fmaf_rn(__fmul_rn(1.f - a.adam.beta2, gi), gi, __fmul_rn(a.adam.beta2, a.v[i]));
    a.m[i] = mi;
    a.v[i] = vi;
    const float mh = mi / a.adam.corr1, vh = vi / a.adam.corr2;
    a.P[i] -= a.adam.lr * mh / (sqrtf(vh) + a.adam.eps);
}

constexpr uint32_t kGradI = 4, kGradJ = 8;   // weights per warp: one per lane
constexpr uint32_t kGradRows = kGradI + kGradJ;
constexpr int kGradStages = 8;
constexpr uint32_t kGradSpan = 2 * kTile;             // samples per stage
constexpr uint32_t kGradPitch = kGradSpan * 4 + 16;   // bytes: eight rows on eight bank groups

__host__ __device__ constexpr uint32_t tiles_of(uint32_t n, uint32_t t) { return (n + t - 1) / t; }

// blocks of grads_kernel: tiles of W2, W1 and W3, then a bias each
__host__ __device__ __forceinline__ uint32_t grad_blocks(uint32_t in, uint32_t h1, uint32_t h2) {
    return tiles_of(h1, kGradI) * tiles_of(h2, kGradJ) + tiles_of(in, kGradI) * tiles_of(h1, kGradJ) +
           tiles_of(h2, kGradI) + h1 + h2 + 1;
}

// Every parameter's gradient, one warp per block.  A weight's gradient is one
// lane's FMA chain over the samples in order (so the sum does not depend on the
// grid), and the chain is the bound: 4 cycles per sample, 8 us for 4096
// (measured: 14).  The warp's 4 + 8 activation rows come through a ring of eight
// 64-sample stages by cp.async.  A bias is the column sum of its layer's
// gradient: 256 strided partial sums, then a tree.  The same lane then makes the
// parameter's Adam update.  Before (GEMM kernels of 4 blocks over 4096 samples,
// column sums, Adam: 16 launches): 860 us per step of 4096 samples for 32 ->
// 64 -> 64 -> 1, now 31 us back to back (34 in a run of four epochs of 64 steps, 41 in
// one epoch, with its statistics, its sample order and its losses).
__global__ void __launch_bounds__(32) grads_kernel(GradArgs a) {
    __shared__ __align__(16) uint8_t ring[kGradStages][kGradRows * kGradPitch];
    const uint32_t lane = threadIdx.x;
    uint32_t b = blockIdx.x;
    const uint32_t nw2 = tiles_of(a.h1, kGradI) * tiles_of(a.h2, kGradJ);
    const uint32_t nw1 = tiles_of(a.in, kGradI) * tiles_of(a.h1, kGradJ);
    const uint32_t nw3 = tiles_of(a.h2, kGradI);
    if (b < nw2 + nw1 + nw3) {
        const float *left, *right;   // gradient (i, j) = left row i . right row j
        uint32_t ni, nj, at;         // rows of each, parameter of (0, 0)
        if (b < nw2) {
            left = a.w.a1, right = a.w.d2, ni = a.h1, nj = a.h2, at = a.L.W2;
        } else if (b < nw2 + nw1) {
            left = a.w.xn, right = a.w.d1, ni = a.in, nj = a.h1, at = a.L.W1, b -= nw2;
        } else {
            left = a.w.a2, right = a.w.dy, ni = a.h2, nj = 1, at = a.L.W3, b -= nw2 + nw1;
        }
        const uint32_t tj = tiles_of(nj, kGradJ);
        const uint32_t i0 = b / tj * kGradI, j0 = b % tj * kGradJ;
        const uint32_t stages = tiles_of(a.n, kGradSpan), tiles = tiles_of(a.n, kTile);
        // this lane's pieces (16 bytes) of a stage's rows; rows past the end:
        // the last row again
        constexpr int kPieces = kGradRows * kGradSpan / 4 / 32;
        const float* src[kPieces];
        uint32_t dst[kPieces];
#pragma unroll
        for (int u = 0; u < kPieces; ++u) {
            const uint32_t piece = lane + 32 * u, r = piece / 16, c = piece % 16;
            src[u] = (r < kGradI ? left + (size_t)min(i0 + r, ni - 1) * a.w.pitch
                                 : right + (size_t)min(j0 + r - kGradI, nj - 1) * a.w.pitch) +
                     c * 4;
            dst[u] = (uint32_t)__cvta_generic_to_shared(&ring[0][r * kGradPitch + c * 16]);
        }
        auto issue = [&](uint32_t s) {
            if (s < stages) {
                const uint32_t st = s % kGradStages * (kGradRows * kGradPitch);
#pragma unroll
                for (int u = 0; u < kPieces; ++u) cp_async16(dst[u] + st, src[u] + s * kGradSpan);
            }
            cp_async_commit();
        };
        for (uint32_t s = 0; s < kGradStages - 1; ++s) issue(s);
        const uint32_t li = lane / kGradJ, lj = lane % kGradJ;
        // the next 32 samples' values are read into registers between the links
        // of the chain over these
        float4 x[2][kTile / 4], y[2][kTile / 4];
        auto landed = [&](uint32_t s) {   // stage s is in; refill the one read before it
            cp_async_wait<kGradStages - 2>();
            __syncwarp();
            issue(s + kGradStages - 1);
        };
        auto fetch = [&](uint32_t t, uint32_t q, int r) {   // tile t is half a stage
            const uint8_t* st = ring[t / 2 % kGradStages] + t % 2 * (kTile * 4) + 16 * q;
            x[r][q] = *reinterpret_cast<const float4*>(st + li * kGradPitch);
            y[r][q] = *reinterpret_cast<const float4*>(st + (kGradI + lj) * kGradPitch);
        };
        float acc = 0.f;
        auto run = [&](uint32_t t, int r) {   // the chain over tile t, held in x[r], y[r]
#pragma unroll
            for (uint32_t q = 0; q < kTile / 4; ++q) {
                fetch(t + 1, q, 1 - r);
                acc = fmaf(x[r][q].x, y[r][q].x, acc);
                acc = fmaf(x[r][q].y, y[r][q].y, acc);
                acc = fmaf(x[r][q].z, y[r][q].z, acc);
                acc = fmaf(x[r][q].w, y[r][q].w, acc);
            }
        };
        landed(0);
#pragma unroll
        for (uint32_t q = 0; q < kTile / 4; ++q) fetch(0, q, 0);
        for (uint32_t t = 0; t < tiles; t += 2) {
            run(t, 0);
            if (t + 1 == tiles) break;
            landed(t / 2 + 1);
            run(t + 1, 1);
        }
        cp_async_wait<0>();
        if (i0 + li < ni && j0 + lj < nj) take_gradient(a, at + (i0 + li) * nj + j0 + lj, acc);
        return;
    }
    b -= nw2 + nw1 + nw3;
    const float* row;
    uint32_t at;
    if (b < a.h2) {
        row = a.w.d2 + (size_t)b * a.w.pitch, at = a.L.b2 + b;
    } else if (b < a.h2 + a.h1) {
        row = a.w.d1 + (size_t)(b - a.h2) * a.w.pitch, at = a.L.b1 + b - a.h2;
    } else {
        row = a.w.dy, at = a.L.b3;
    }
    // partial sum p = entries p, p + 256, ...; then red[p] += red[p + w] for
    // w = 128 .. 1 (lane: partial sums lane + 32 u)
    float red[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) red[u] = 0.f;
#pragma unroll 4
    for (uint32_t m = 0; m < a.n; m += 256)
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const uint32_t e = m + lane + 32 * u;
            red[u] += e < a.n ? row[e] : 0.f;
        }
#pragma unroll
    for (int w = 4; w > 0; w >>= 1)
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (u < w) red[u] += red[u + w];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) red[0] += __shfl_down_sync(0xffffffffu, red[0], o);
    if (lane == 0) take_gradient(a, at, red[0]);
}

// the batch's loss from its tiles' partial sums
__global__ void loss_kernel(const float* __restrict__ part, uint32_t tiles,
                            float* __restrict__ loss) {
    float l = 0.f;
    for (uint32_t i = threadIdx.x; i < tiles; i += 32) l += part[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (threadIdx.x == 0) *loss = l;
}

__global__ void to_bf16_kernel(const float* __restrict__ src, __nv_bfloat16* __restrict__ dst,
                               uint32_t n) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dst[i] = __float2bfloat16_rn(src[i]);
}

// the layers over n samples (rows perm[i] of x and t when perm is set):
// outputs into y, or with y null a training step's activations into M->work
int launch_layers(hc_mlp* M, const float* x, const float* t, const uint32_t* perm, uint32_t n,
                  float* y, cudaStream_t s) {
    if (allow_shared(layers_kernel, sizeof(LayerSmem)) != cudaSuccess) return HC_ERR_CUDA;
    const LayerArgs a{layout_of(M->in, M->h1, M->h2), M->params, M->in, M->h1, M->h2, n, x, t,
                      perm, y, work_of(M)};
    layers_kernel<<<tiles_of(n, kTile), 256, sizeof(LayerSmem), s>>>(a);
    count_launches(1);
    return cudaGetLastError() == cudaSuccess ? HC_OK : HC_ERR_CUDA;
}

// gradients of the batch whose activations are in M->work into M->grads (and
// the Adam step, when given)
int launch_grads(hc_mlp* M, uint32_t n, const Adam* adam, cudaStream_t s) {
    const GradArgs a{layout_of(M->in, M->h1, M->h2), M->in, M->h1, M->h2, n, work_of(M),
                     M->params, M->grads, M->adam_m, M->adam_v, adam != nullptr,
                     adam ? *adam : Adam{}};
    grads_kernel<<<grad_blocks(M->in, M->h1, M->h2), 32, 0, s>>>(a);
    count_launches(1);
    return cudaGetLastError() == cudaSuccess ? HC_OK : HC_ERR_CUDA;
}

// M->loss of the batch whose activations are in M->work
int launch_loss(hc_mlp* M, uint32_t n, cudaStream_t s) {
    loss_kernel<<<1, 32, 0, s>>>(work_of(M).loss, tiles_of(n, kTile), M->loss);
    count_launches(1);
    return cudaGetLastError() == cudaSuccess ? HC_OK : HC_ERR_CUDA;
}

int read_loss(hc_mlp* M, uint32_t n, float* loss_host, cudaStream_t s) {
    if (int rc = launch_loss(M, n, s)) return rc;
    if (cudaMemcpyAsync(loss_host, M->loss, sizeof(float), cudaMemcpyDeviceToHost, s) !=
            cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return HC_ERR_CUDA;
    return HC_OK;
}

int refresh_bf16(hc_mlp* M, cudaStream_t s) {
    if (!M->bf_stale) return HC_OK;
    const Layout L = layout_of(M->in, M->h1, M->h2);
    const uint32_t n1 = M->in * M->h1, n2 = M->h1 * M->h2, n3 = M->h2;
    to_bf16_kernel<<<(n1 + 255) / 256, 256, 0, s>>>(M->params + L.W1, M->wbf, n1);
    to_bf16_kernel<<<(n2 + 255) / 256, 256, 0, s>>>(M->params + L.W2, M->wbf + n1, n2);
    to_bf16_kernel<<<(n3 + 255) / 256, 256, 0, s>>>(M->params + L.W3, M->wbf + n1 + n2, n3);
    count_launches(3);
    M->bf_stale = false;
    return cudaGetLastError() == cudaSuccess ? HC_OK : HC_ERR_CUDA;
}

// ---------------------------------------------------------- inference
constexpr int kPredWarps = 8;

struct MlpView {
    uint32_t in, h1, h2;
    const __nv_bfloat16* wbf;   // W1 | W2 | W3
    const float* params;        // for b1 b2 b3 mu isd
    Layout L;
};

__device__ __forceinline__ float bf(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// y of G samples whose raw features sit in xs[i * G + g] (warp-shared memory).
// Weights in shared memory (bf16), inputs of each layer rounded to bf16,
// accumulation in float32, inputs ascending.  Lane j computes hidden units j and
// j + 32 of all G samples: a weight is read and widened once for them, and an
// input of all of them is one load (G = 4: 13 instructions for 8 FMAs; one
// sample and one unit at a time took 4 for each).  UNITS = 1: layers of at most 32
// units (8 -> 8 for 4M samples: 1.08 ms with the second unit computed all the same,
// 0.90 without).
template <int G, int UNITS>
__device__ __forceinline__ void mlp_units(const __nv_bfloat16* w, uint32_t in, uint32_t out,
                                          const float* xs, int lane, float (&acc)[2][G]) {
    const __nv_bfloat16* w0 = w + min((uint32_t)lane, out - 1);
    const __nv_bfloat16* w1 = w + min((uint32_t)lane + 32, out - 1);
#pragma unroll 4
    for (uint32_t i = 0; i < in; ++i) {
        const float v0 = __bfloat162float(w0[i * out]);
        const float v1 = UNITS > 1 ? __bfloat162float(w1[i * out]) : 0.f;
        float x[G];
        if constexpr (G == 4)
            *reinterpret_cast<float4*>(x) = *reinterpret_cast<const float4*>(xs + 4 * i);
        else
#pragma unroll
            for (int g = 0; g < G; ++g) x[g] = xs[i * G + g];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            acc[0][g] = fmaf(x[g], v0, acc[0][g]);
            if constexpr (UNITS > 1) acc[1][g] = fmaf(x[g], v1, acc[1][g]);
        }
    }
}

template <int G>
__device__ __forceinline__ void mlp_layer(const __nv_bfloat16* w, uint32_t in, uint32_t out,
                                          const float* xs, int lane, float (&acc)[2][G]) {
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int g = 0; g < G; ++g) acc[u][g] = 0.f;
    if (out > 32)
        mlp_units<G, 2>(w, in, out, xs, lane, acc);
    else
        mlp_units<G, 1>(w, in, out, xs, lane, acc);
}

template <int G>
__device__ void mlp_warp_forward(const MlpView& V, const __nv_bfloat16* sW1,
                                 const __nv_bfloat16* sW2, const __nv_bfloat16* sW3,
                                 const float* sb, float* xs, float* hs, int lane, float (&y)[G]) {
    const float* b1 = sb;
    const float* b2 = sb + kMaxDim;
    const float b3 = sb[2 * kMaxDim];
    const float* mu = sb + 2 * kMaxDim + 1;
    const float* isd = mu + kMaxDim;
    for (uint32_t i = lane; i < V.in; i += 32)
#pragma unroll
        for (int g = 0; g < G; ++g) xs[i * G + g] = bf((xs[i * G + g] - mu[i]) * isd[i]);
    __syncwarp();
    float acc[2][G];
    mlp_layer<G>(sW1, V.in, V.h1, xs, lane, acc);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const uint32_t j = (uint32_t)lane + 32 * u;
        if (j < V.h1)
#pragma unroll
            for (int g = 0; g < G; ++g) hs[j * G + g] = bf(fmaxf(acc[u][g] + b1[j], 0.f));
    }
    __syncwarp();
    mlp_layer<G>(sW2, V.h1, V.h2, hs, lane, acc);
#pragma unroll
    for (int g = 0; g < G; ++g) y[g] = 0.f;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const uint32_t j = (uint32_t)lane + 32 * u;
        if (j < V.h2)
#pragma unroll
            for (int g = 0; g < G; ++g)
                y[g] = fmaf(bf(fmaxf(acc[u][g] + b2[j], 0.f)), __bfloat162float(sW3[j]), y[g]);
    }
#pragma unroll
    for (int g = 0; g < G; ++g) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) y[g] += __shfl_xor_sync(0xffffffffu, y[g], o);
        y[g] += b3;
    }
    __syncwarp();
}

// Stages bf16 weights and float biases / normalisation in shared memory.
__device__ void stage_weights(const MlpView& V, __nv_bfloat16* sW, float* sb) {
    const uint32_t nw = V.in * V.h1 + V.h1 * V.h2 + V.h2;
    for (uint32_t i = threadIdx.x; i < nw; i += blockDim.x) sW[i] = V.wbf[i];
    for (uint32_t i = threadIdx.x; i < 4 * kMaxDim + 1; i += blockDim.x) {
        float v = 0.f;
        if (i < kMaxDim) v = i < V.h1 ? V.params[V.L.b1 + i] : 0.f;
        else if (i < 2 * kMaxDim) v = i - kMaxDim < V.h2 ? V.params[V.L.b2 + i - kMaxDim] : 0.f;
        else if (i == 2 * kMaxDim) v = V.params[V.L.b3];
        else if (i < 3 * kMaxDim + 1) {
            const uint32_t j = i - 2 * kMaxDim - 1;
            v = j < V.in ? V.params[V.L.mu + j] : 0.f;
        } else {
            const uint32_t j = i - 3 * kMaxDim - 1;
            v = j < V.in ? V.params[V.L.isd + j] : 1.f;
        }
        sb[i] = v;
    }
    __syncthreads();
}

__global__ void __launch_bounds__(kPredWarps * 32) mlp_infer_kernel(MlpView V,
                                                                    const float* __restrict__ x,
                                                                    uint32_t n, float* __restrict__ y) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __nv_bfloat16* sW = reinterpret_cast<__nv_bfloat16*>(smem_raw);
    const uint32_t nw = V.in * V.h1 + V.h1 * V.h2 + V.h2;
    float* sb = reinterpret_cast<float*>(smem_raw + ((nw * 2 + 15) & ~15u));
    float* sx = sb + 4 * kMaxDim + 1 + 3;
    stage_weights(V, sW, sb);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float* xs = sx + warp * 2 * kMaxDim;
    float* hs = xs + kMaxDim;
    for (uint32_t i = blockIdx.x * kPredWarps + warp; i < n; i += gridDim.x * kPredWarps) {
        for (uint32_t j = lane; j < V.in; j += 32) xs[j] = x[(size_t)i * V.in + j];
        __syncwarp();
        float yi[1];
        mlp_warp_forward<1>(V, sW, sW + V.in * V.h1, sW + V.in * V.h1 + V.h1 * V.h2, sb, xs, hs,
                            lane, yi);
        if (lane == 0) y[i] = yi[0];
        __syncwarp();
    }
}

size_t pred_smem(uint32_t in, uint32_t h1, uint32_t h2, int G = 1) {
    const uint32_t nw = in * h1 + h1 * h2 + h2;
    return ((nw * 2 + 15) & ~15u) + sizeof(float) * (4 * kMaxDim + 1 + 3) +
           sizeof(float) * kPredWarps * 2 * kMaxDim * G + sizeof(uint32_t) * kPredWarps * (64 + 128);
}

// ------------------------------------------------------------ features
// Octave encoding: 0 for g = 0, else 1 + e + f / 65536 with e the top set bit
// of the 128-bit g and f the 16 bits below it.  Exact in float32.
__device__ __forceinline__ float octave128(uint64_t hi, uint64_t lo) {
    if (!hi && !lo) return 0.f;
    const int e = hi ? 127 - __clzll((long long)hi) : 63 - __clzll((long long)lo);
    const unsigned __int128 g = ((unsigned __int128)hi << 64) | lo;
    const uint32_t f = e >= 16 ? (uint32_t)(g >> (e - 16)) & 0xFFFFu
                               : (uint32_t)(g << (16 - e)) & 0xFFFFu;
    return 1.0f + (float)e + (float)f * (1.0f / 65536.0f);
}

constexpr float kFeatNone = 130.0f;

// 128-bit gap (a - b) of two keys, octave-encoded
__device__ __forceinline__ float key_gap_octave(uint64_t ah, uint64_t al, uint64_t bh, uint64_t bl) {
    const uint64_t gl = al - bl, gh = ah - bh - (al < bl ? 1u : 0u);
    return octave128(gh, gl);
}

// Whether the low words of two keys whose high words differ by dh cannot show in
// the octave of their gap: its top bit and the 16 below lie in dh, above bits of
// dh that are not all zero, so a borrow from the low words ends below them.  Holds
// for all but one gap in thousands of a long list, whose low word (the row's key
// where the index keeps high words only) is then not computed.
__device__ __forceinline__ bool gap_from_high(uint64_t dh) {
    const int e = 63 - __clzll((long long)dh);
    return e > 16 && (dh & ((1ull << (e - 16)) - 1));
}

// The 4 * curves features of one query into xs (warp-shared, feature i at
// xs[i * stride]), from the positions pos_w of lists 0..curves-1 (khi/klo: lane c holds curve c's key).
// All curves at once: the 8-entry centre windows fill 32-row steps (slot
// 8 c + j = entry j of curve c's window, distances parked in sd), and lanes
// 2 c, 2 c + 1 take curve c's predecessor and successor gaps (a low key word
// recomputed from its row where the index keeps high words only).
__device__ void query_features(const IndexView& ix, const uint8_t* qrow, uint4 qv0,
                               const uint32_t* pos_w, uint64_t khi, uint64_t klo, float* xs,
                               uint32_t* sd, int lane, uint32_t stride = 1) {
    const uint8_t* db = static_cast<const uint8_t*>(ix.db);
    const uint32_t C = ix.P.curves;
    // the loads of the gaps first: lanes 2c, 2c + 1 the predecessor and the
    // successor of curve c's key
    const uint32_t gc = (uint32_t)lane / 2 < C ? (uint32_t)lane / 2 : 0u;
    bool near = (uint32_t)lane / 2 < C;
    uint64_t ge = 0, gh = 0;
    {
        const uint64_t off = ix.list_off[gc];
        const uint32_t n = (uint32_t)(ix.list_off[gc + 1] - off), pos = pos_w[gc];
        near = near && ((lane & 1) ? pos < n : pos > 0);
        ge = off + pos - ((lane & 1) ? 0 : 1);
        if (near) gh = ix.keys_hi[ge];
    }
    // centre window of curve c = lane / 8 (per slot)
    for (uint32_t t = 0; t < C; t += 4) {
        const uint32_t c = t + (uint32_t)lane / 8, j = (uint32_t)lane % 8;
        uint32_t id = 0;
        bool valid = false;
        if (c < C) {
            const uint64_t off = ix.list_off[c];
            const uint32_t n = (uint32_t)(ix.list_off[c + 1] - off);
            const uint32_t pos = pos_w[c];
            const uint32_t lo = pos > 4 ? pos - 4 : 0u, hi = pos + 4 < n ? pos + 4 : n;
            valid = lo + j < hi;
            if (valid) id = __ldg(ix.ids + off + lo + j);
            if (!HC_IN_BOUNDS(kSiteRow, id, ix.rows)) id = 0u;
        }
        uint64_t cands[ChunkWidth<8>::NG];
        chunk_candidates_n<false, 8>(db, ix.row_bytes, qrow, qv0, id, 32u, lane, cands);
        // lane l holds the row (l % 8) * 4 + l / 8 of the step
        const uint32_t r = ((uint32_t)lane % 8) * 4 + (uint32_t)lane / 8;
        const bool rvalid = __shfl_sync(0xffffffffu, valid, (int)r);
        sd[8 * t + r] = rvalid ? (uint32_t)(cands[0] >> 32) : 0xFFFFFFFFu;
    }
    __syncwarp();
    float f0 = kFeatNone, f1 = kFeatNone, f2 = kFeatNone, f3 = kFeatNone;
    {
        const uint64_t kh = __shfl_sync(0xffffffffu, khi, (int)gc);
        const uint64_t kl = __shfl_sync(0xffffffffu, klo, (int)gc);
        float gap = kFeatNone;
        if (near) {
            const uint64_t dh = (lane & 1) ? gh - kh : kh - gh;
            if (gap_from_high(dh)) {
                gap = octave128(dh, 0);
            } else {
                const uint64_t gl = entry_key_lo(ix, gc, ge);
                gap = (lane & 1) ? key_gap_octave(gh, gl, kh, kl) : key_gap_octave(kh, kl, gh, gl);
            }
        }
        const float other = __shfl_xor_sync(0xffffffffu, gap, 1);
        f0 = (lane & 1) ? other : gap;
        f1 = (lane & 1) ? gap : other;
    }
    if ((uint32_t)lane < C) {
        // centre-window distances of curve lane
        uint32_t dmin = 0xFFFFFFFFu, cnt = 0;
        uint64_t dsum = 0;
        for (uint32_t j = 0; j < 8; ++j) {
            const uint32_t v = sd[8 * lane + j];
            if (v != 0xFFFFFFFFu) {
                dmin = min(dmin, v);
                dsum += v;
                ++cnt;
            }
        }
        if (cnt) {
            f2 = octave128(0, dmin);
            f3 = octave128(0, dsum / cnt);
        }
    }
    // lane c < C gathers its curve's gap pair from lane 2c
    const float g0 = __shfl_sync(0xffffffffu, f0, (2 * lane) & 31);
    const float g1 = __shfl_sync(0xffffffffu, f1, (2 * lane) & 31);
    if ((uint32_t)lane < C) {
        xs[(4 * lane + 0) * stride] = g0;
        xs[(4 * lane + 1) * stride] = g1;
        xs[(4 * lane + 2) * stride] = f2;
        xs[(4 * lane + 3) * stride] = f3;
    }
    __syncwarp();
}

__device__ __forceinline__ void warp_keys_positions(const IndexView& ix, const uint8_t* qrow,
                                                    uint32_t* pos_w, uint64_t& khi, uint64_t& klo,
                                                    int lane) {
    khi = 0;
    klo = 0;
    const uint32_t curves = ix.P.curves;
    if ((uint32_t)lane < curves) curve_key_call(qrow, ix.P, (uint32_t)lane, khi, klo);
    if ((uint32_t)lane < curves) {
        const uint64_t off = ix.list_off[lane];
        const uint32_t n = (uint32_t)(ix.list_off[lane + 1] - off);
        pos_w[lane] = lower_bound_key(ix, (uint32_t)lane, off, n, khi, klo);
    }
    __syncwarp();
}

__global__ void __launch_bounds__(kPredWarps * 32) features_kernel(IndexView ix, const uint8_t* q,
                                                                   uint32_t nq, float* feat) {
    __shared__ uint32_t s_pos[kPredWarps][64 + 128];   // positions, then window distances
    __shared__ float s_x[kPredWarps][4 * 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t qi = blockIdx.x * kPredWarps + warp;
    if (qi >= nq) return;
    const uint8_t* qrow = q + (size_t)qi * ix.row_bytes;
    uint64_t khi, klo;
    warp_keys_positions(ix, qrow, s_pos[warp], khi, klo, lane);
    const uint32_t s = (uint32_t)lane % 8;
    const uint4 qv0 = s < (ix.row_bytes >> 4) ? ldg16(qrow + s * 16) : make_uint4(0, 0, 0, 0);
    query_features(ix, qrow, qv0, s_pos[warp], khi, klo, s_x[warp], s_pos[warp] + 64, lane);
    for (uint32_t j = lane; j < 4 * ix.P.curves; j += 32)
        feat[(size_t)qi * 4 * ix.P.curves + j] = s_x[warp][j];
}

// features -> MLP -> p = clamp(ceil(2^(y + margin)), p_lo, p_hi), per query.
// A warp takes G queries at once (at most 32 / G curves): lane g * 32 / G + c
// computes curve c's key and position of query g, so that the keys and the
// dependent loads of the searches, which fill `curves` lanes for one query, are
// done for all of them together, and the layers read every weight once.  Bound by
// the latency of scattered loads (long scoreboard half of the stalls, 45% of the
// issue slots): of 590 us for 100,000 queries on 10M rows and 8 curves the searches
// are 265, the keys 146, the 64 rows of each query's features 143, the layers 65;
// one query per warp, every gap's low word computed: 1,025 us.
template <int G>
__global__ void __launch_bounds__(kPredWarps * 32, 4) predict_depths_kernel(
    IndexView ix, MlpView V, const uint8_t* q, uint32_t nq, float margin, uint32_t p_lo,
    uint32_t p_hi, uint32_t* p_out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __nv_bfloat16* sW = reinterpret_cast<__nv_bfloat16*>(smem_raw);
    const uint32_t nw = V.in * V.h1 + V.h1 * V.h2 + V.h2;
    float* sb = reinterpret_cast<float*>(smem_raw + ((nw * 2 + 15) & ~15u));
    float* sx = sb + 4 * kMaxDim + 1 + 3;
    uint32_t* spos = reinterpret_cast<uint32_t*>(sx + kPredWarps * 2 * kMaxDim * G);
    stage_weights(V, sW, sb);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float* xs = sx + warp * 2 * kMaxDim * G;
    float* hs = xs + kMaxDim * G;
    uint32_t* pos_w = spos + warp * (64 + 128);
    constexpr int kLanes = 32 / G;   // per query
    const uint32_t c = (uint32_t)lane % kLanes, s = (uint32_t)lane % 8;
    for (uint64_t q0 = ((uint64_t)blockIdx.x * kPredWarps + warp) * G; q0 < nq;
         q0 += (uint64_t)gridDim.x * kPredWarps * G) {
        const uint32_t n = (uint32_t)min((uint64_t)G, nq - q0);
        uint64_t khi = 0, klo = 0;
        if (c < ix.P.curves && (uint32_t)lane / kLanes < n) {
            curve_key_call(q + (size_t)(q0 + lane / kLanes) * ix.row_bytes, ix.P, c, khi, klo);
            const uint64_t off = ix.list_off[c];
            pos_w[lane] = lower_bound_key(ix, c, off, (uint32_t)(ix.list_off[c + 1] - off), khi,
                                          klo);
        }
        __syncwarp();
        for (uint32_t g = 0; g < n; ++g) {
            const uint8_t* qrow = q + (size_t)(q0 + g) * ix.row_bytes;
            const uint4 qv0 =
                s < (ix.row_bytes >> 4) ? ldg16(qrow + s * 16) : make_uint4(0, 0, 0, 0);
            const int from = (int)(g * kLanes + c);
            const uint64_t kh = __shfl_sync(0xffffffffu, khi, from);
            const uint64_t kl = __shfl_sync(0xffffffffu, klo, from);
            query_features(ix, qrow, qv0, pos_w + g * kLanes, kh, kl, xs + g, pos_w + 64, lane, G);
        }
        float y[G];
        mlp_warp_forward<G>(V, sW, sW + V.in * V.h1, sW + V.in * V.h1 + V.h1 * V.h2, sb, xs, hs,
                            lane, y);
#pragma unroll
        for (int g = 0; g < G; ++g)
            if (lane == g && g < n) {
                const float e = fminf(fmaxf(y[g] + margin, -1.0f), 30.0f);
                uint32_t p = (uint32_t)ceilf(exp2f(e));
                p = p < p_lo ? p_lo : (p > p_hi ? p_hi : p);
                p_out[q0 + g] = p;
            }
        __syncwarp();
    }
}

template <int G>
cudaError_t go_predict(const IndexView& ix, const MlpView& V, const void* q, uint32_t nq,
                       float margin, uint32_t p_lo, uint32_t p_hi, uint32_t* p_out, int sms,
                       cudaStream_t s) {
    const size_t smem = pred_smem(V.in, V.h1, V.h2, G);
    const cudaError_t e =
        allow_shared(predict_depths_kernel<G>, pred_smem(kMaxDim, kMaxDim, kMaxDim, G));
    if (e != cudaSuccess) return e;
    const uint32_t per = kPredWarps * G;
    const unsigned blocks =
        std::min((uint32_t)(((uint64_t)nq + per - 1) / per), (uint32_t)sms * 8);
    predict_depths_kernel<G><<<blocks, kPredWarps * 32, smem, s>>>(
        ix, V, static_cast<const uint8_t*>(q), nq, margin, p_lo, p_hi, p_out);
    count_launches(1);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- labels
// The windows of a query are nested in p, so the top-k at depth p equals the
// top-k at p_max once every neighbour of the latter lies in some window of depth
// p: the label is the largest, over those neighbours, of the smallest depth at
// which any list holds it.  One warp per query (in the batch's key order, whose
// neighbours share lines of the lists) holds the neighbours in registers, entry
// r 32 + lane in t[r] of the lane, and streams the ids of its windows past a
// 2048-bit filter of them; the few ids that pass are compared with all: about
// ten instructions per 32 ids, no row is read.  50,000 queries at p_max = 512 on
// 10M rows and 8 lists: 4.8 ms, nearly all of it the one walk at p_max, against
// 82.4 ms for a binary search over p (eleven walks).
constexpr int kLabelWarps = 8;
constexpr uint32_t kLabelSlice = 1u << 17;   // queries labelled at once
constexpr uint32_t kFilterBits = 2048;

template <int KR>
__global__ void __launch_bounds__(kLabelWarps * 32) label_kernel(
    IndexView ix, uint32_t nq, uint32_t k, uint32_t p_max, const int32_t* __restrict__ ref,
    const uint32_t* __restrict__ order, const uint32_t* __restrict__ pos_cm,
    uint32_t* __restrict__ out) {
    __shared__ uint32_t filters[kLabelWarps][kFilterBits / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t w = blockIdx.x * kLabelWarps + warp;
    if (w >= nq) return;
    const uint32_t qi = __ldg(order + w);
    if (!HC_IN_BOUNDS(kSiteQuery, qi, nq)) return;
    uint32_t* filter = filters[warp];
    auto slot = [](uint32_t id) { return (id * 2654435761u) >> 21; };
    for (uint32_t i = lane; i < kFilterBits / 32; i += 32) filter[i] = 0;
    __syncwarp();
    uint32_t t[KR], depth[KR];   // 0xFFFFFFFF: no neighbour (ids are below 2^31)
#pragma unroll
    for (int r = 0; r < KR; ++r) {
        const uint32_t e = r * 32 + lane;
        t[r] = e < k ? (uint32_t)__ldg(ref + (size_t)qi * k + e) : 0xFFFFFFFFu;
        depth[r] = t[r] == 0xFFFFFFFFu ? 0u : 0xFFFFFFFFu;
        if (t[r] != 0xFFFFFFFFu) atomicOr(&filter[slot(t[r]) / 32], 1u << (slot(t[r]) % 32));
    }
    __syncwarp();
    const uint32_t curves = ix.P.curves, parts = ix.lists / curves;
    for (uint32_t L = 0; L < ix.lists; ++L) {
        const uint64_t off = ix.list_off[L];
        const uint32_t n = (uint32_t)(ix.list_off[L + 1] - off);
        const uint32_t pos =
            __ldg(pos_cm + (size_t)qi * ix.lists + (L % curves) * parts + L / curves);
        const uint32_t lo = pos > p_max ? pos - p_max : 0u;
        const uint32_t hi = (uint64_t)pos + p_max < (uint64_t)n ? pos + p_max : n;
        if (!HC_IN_BOUNDS(kSiteWindow, hi, (uint64_t)n + 1)) continue;
        constexpr int U = 4;   // loads in flight
        for (uint32_t base = lo; base < hi; base += 32 * U) {
            uint32_t id[U];
            bool ok[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t e = base + 32 * u + (uint32_t)lane;
                ok[u] = e < hi;
                id[u] = ok[u] ? __ldg(ix.ids + off + e) : 0u;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t s = slot(id[u]);
                uint32_t hit = __ballot_sync(0xffffffffu, ok[u] && (filter[s / 32] >> (s % 32) & 1u));
                while (hit) {
                    const int src = __ffs(hit) - 1;
                    hit &= hit - 1;
                    const uint32_t x = __shfl_sync(0xffffffffu, id[u], src);
                    const uint32_t e = base + 32 * u + (uint32_t)src;
                    const uint32_t d = e >= pos ? e - pos + 1 : pos - e;
#pragma unroll
                    for (int r = 0; r < KR; ++r)
                        if (t[r] == x) depth[r] = min(depth[r], d);
                }
            }
        }
    }
    uint32_t label = 0;
#pragma unroll
    for (int r = 0; r < KR; ++r) label = max(label, depth[r]);
    label = __reduce_max_sync(0xffffffffu, label);
    if (lane == 0) out[qi] = label;
}

MlpView view_of_mlp(const hc_mlp* M) {
    MlpView V;
    V.in = M->in;
    V.h1 = M->h1;
    V.h2 = M->h2;
    V.wbf = M->wbf;
    V.params = M->params;
    V.L = layout_of(M->in, M->h1, M->h2);
    return V;
}

bool dev_ptr(const void* p) {
    if (!p) return false;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

int features_ok(const hc_index* idx) {
    if (!idx) return HC_ERR_ARG;
    if (idx->params.dtype != HC_U8 || idx->params.partitions != 1) return HC_ERR_ARG;
    if (idx->params.curves > 16 || idx->row_bytes > 8 * 16 * 32) return HC_ERR_ARG;
    return HC_OK;
}

// -------------------------------------------------------------- training
// regression target of a depth label: log2(max(label, 1))
__global__ void fit_targets_kernel(const uint32_t* __restrict__ labels, uint32_t n,
                                   float* __restrict__ t) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) t[i] = log2f((float)(labels[i] > 1u ? labels[i] : 1u));
}

// Feature statistics: mean, then the unbiased standard deviation about it
// (two passes, float64 sums); mu = mean, isd = 1 / max(sd, 1e-3).  A column's sum
// is 256 strided partial sums (sample i in partial i % 256), added up 32 at a
// time by a butterfly and then in order.  A block is one warp: 32 partials of one
// column, a lane per partial, 16 loads in flight per lane (the other columns of a
// 32-byte sector come from L2: blocks of one g run side by side); sums[c][g]: the sum
// of partials 32 g .. of column c (pass 1: of x, pass 2: of (x - mean)^2).
constexpr uint32_t kStatGroups = 8;   // of 32 partial sums
__device__ __forceinline__ double stat_total(const double* s) {
    double t = 0.0;
    for (uint32_t g = 0; g < kStatGroups; ++g) t += s[g];
    return t;
}

template <bool SQUARES>
__global__ void __launch_bounds__(32) fit_stats_kernel(const float* __restrict__ x, uint32_t n,
                                                        uint32_t in, double* __restrict__ sums,
                                                        double* __restrict__ squares) {
    const uint32_t lane = threadIdx.x, c = blockIdx.x, g = blockIdx.y;
    const double mean = SQUARES ? stat_total(sums + c * kStatGroups) / (double)n : 0.0;
    double acc = 0.0;
#pragma unroll 1
    for (uint64_t i = g * 32 + lane; i < n; i += 256 * 16) {
        float v[16];
#pragma unroll
        for (int u = 0; u < 16; ++u)
            v[u] = i + 256ull * u < n ? __ldg(x + (i + 256ull * u) * in + c) : 0.f;
#pragma unroll
        for (int u = 0; u < 16; ++u)
            if (i + 256ull * u < n) {
                const double d = SQUARES ? (double)v[u] - mean : (double)v[u];
                acc += SQUARES ? d * d : d;
            }
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) (SQUARES ? squares : sums)[c * kStatGroups + g] = acc;
}

__global__ void fit_norm_kernel(uint32_t n, uint32_t in, const double* __restrict__ sums,
                                const double* __restrict__ squares, float* __restrict__ mu,
                                float* __restrict__ isd) {
    const uint32_t c = threadIdx.x;
    if (c >= in) return;
    const double sd = n > 1 ? sqrt(stat_total(squares + c * kStatGroups) / (double)(n - 1)) : 0.0;
    mu[c] = (float)(stat_total(sums + c * kStatGroups) / (double)n);
    isd[c] = (float)(1.0 / (sd > 1e-3 ? sd : 1e-3));
}

// SplitMix64 (Steele, Lea and Flood, OOPSLA 2014) of a counter
__device__ __forceinline__ uint64_t splitmix64(uint64_t z) {
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// random 32-bit sort keys of epoch e: the order of the samples in that epoch
__global__ void fit_keys_kernel(uint64_t seed, uint32_t epoch, uint32_t n,
                                uint64_t* __restrict__ keys) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n)
        keys[i] = splitmix64(seed ^ ((uint64_t)epoch << 40) ^ (uint64_t)i) >> 32;
}

}  // namespace

// predictor launch used by the serving loop (serve.cu)
namespace hc {
int mlp_prepare_inference(hc_mlp* M, const hc_index* idx, cudaStream_t s) {
    if (!M || !idx || M->in != 4 * idx->params.curves) return HC_ERR_ARG;
    if (int rc = refresh_bf16(M, s)) return rc;
    return cudaStreamSynchronize(s) == cudaSuccess ? HC_OK : HC_ERR_CUDA;
}

cudaError_t launch_predict_depths(hc_mlp* M, const hc_index* idx, const void* q, uint32_t nq,
                                  float margin, uint32_t p_lo, uint32_t p_hi, uint32_t* p_out,
                                  cudaStream_t s) {
    if (nq == 0) return cudaSuccess;
    if (refresh_bf16(M, s) != HC_OK) return cudaErrorUnknown;
    const MlpView V = view_of_mlp(M);
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const IndexView v = view_of(idx);
    // Queries per warp: more where the warps in flight are full anyway (100,000
    // queries, 8 curves: 854 us at one, 702 at two, 590 at four; 4,096: 65, 63, 70;
    // 8,192: 107, 95, 104; 12,288: 143, 133, 123; 16 curves: 100,000 1,030 at one,
    // 918 at two, but 12,288 176 and 183)
    const uint32_t resident = (uint32_t)sms * 4 * kPredWarps;   // warps
    if (v.P.curves <= 8 && nq >= 2 * resident)
        return go_predict<4>(v, V, q, nq, margin, p_lo, p_hi, p_out, sms, s);
    if (v.P.curves <= 16 && nq >= (v.P.curves <= 8 ? 1 : 6) * resident)
        return go_predict<2>(v, V, q, nq, margin, p_lo, p_hi, p_out, sms, s);
    return go_predict<1>(v, V, q, nq, margin, p_lo, p_hi, p_out, sms, s);
}
}  // namespace hc

extern "C" {

HC_API int hc_features(hc_index* idx, const void* q_dev, uint32_t nq, float* feat_dev,
                       void* cuda_stream) {
    TraceRange tr("hc_features");
    if (int rc = features_ok(idx)) return rc;
    if (nq == 0) return HC_OK;
    if (!dev_ptr(q_dev) || !dev_ptr(feat_dev) || ((uintptr_t)q_dev & 15)) return HC_ERR_ARG;
    features_kernel<<<(nq + kPredWarps - 1) / kPredWarps, kPredWarps * 32, 0,
                      static_cast<cudaStream_t>(cuda_stream)>>>(
        view_of(idx), static_cast<const uint8_t*>(q_dev), nq, feat_dev);
    count_launches(1);
    return cudaGetLastError() == cudaSuccess ? HC_OK : HC_ERR_CUDA;
}

HC_API int hc_probe_labels(hc_index* idx, const void* q_dev, uint32_t nq, uint32_t k,
                           uint32_t p_max, uint32_t* p_min_dev, void* cuda_stream) {
    TraceRange tr("hc_probe_labels");
    if (!idx || k < 1 || k > 128 || p_max > (1u << 30)) return HC_ERR_ARG;
    if (nq == 0) return HC_OK;
    if (!dev_ptr(q_dev) || !dev_ptr(p_min_dev) || ((uintptr_t)q_dev & 15)) return HC_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    if (alloc_should_fail()) return HC_ERR_OOM;
    // slices of the batch bound the scratch: the key-order workspace, then the
    // neighbours at p_max (ids and distances); smaller ones when memory is short
    uint32_t slice = nq < kLabelSlice ? nq : kLabelSlice;
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    char* buf = nullptr;
    size_t ws = 0, res = 0;
    for (;; slice = (slice + 1) / 2) {
        ws = al(ordered_workspace(idx, slice));
        res = al((size_t)slice * k * 4);
        if (cudaMallocAsync((void**)&buf, ws + 2 * res, s) == cudaSuccess) break;
        cudaGetLastError();
        if (slice <= 1024) return HC_ERR_OOM;
    }
    int32_t* ref = reinterpret_cast<int32_t*>(buf + ws);
    const IndexView ix = view_of(idx);
    int rc = HC_OK;
    for (uint32_t q0 = 0; !rc && q0 < nq; q0 += slice) {
        const uint32_t b = nq - q0 < slice ? nq - q0 : slice;
        const uint8_t* q = static_cast<const uint8_t*>(q_dev) + (size_t)q0 * ix.row_bytes;
        if ((rc = ordered_query(idx, q, b, k, p_max, ref, buf + ws + res, buf, s))) break;
        const uint32_t* order = ordered_ranks(idx, b, buf);
        const uint32_t* pos = ordered_positions(idx, b, buf);
        const unsigned g = (b + kLabelWarps - 1) / kLabelWarps;
        if (k <= 32)
            label_kernel<1><<<g, kLabelWarps * 32, 0, s>>>(ix, b, k, p_max, ref, order, pos,
                                                           p_min_dev + q0);
        else
            label_kernel<4><<<g, kLabelWarps * 32, 0, s>>>(ix, b, k, p_max, ref, order, pos,
                                                           p_min_dev + q0);
        count_launches(1);
        if (cudaGetLastError() != cudaSuccess) rc = HC_ERR_CUDA;
    }
    cudaFreeAsync(buf, s);
    return rc;
}

HC_API int hc_mlp_create(uint32_t in_dim, uint32_t hidden1, uint32_t hidden2, uint32_t max_batch,
                         hc_mlp** out) {
    if (!out) return HC_ERR_ARG;
    *out = nullptr;
    if (in_dim < 1 || in_dim > kMaxDim || hidden1 < 1 || hidden1 > kMaxDim || hidden2 < 1 ||
        hidden2 > kMaxDim || max_batch < 1 || max_batch > (1u << 20))
        return HC_ERR_ARG;
    hc_mlp* M = new (std::nothrow) hc_mlp();
    if (!M) return HC_ERR_OOM;
    M->in = in_dim;
    M->h1 = hidden1;
    M->h2 = hidden2;
    M->max_batch = max_batch;
    const Layout L = layout_of(in_dim, hidden1, hidden2);
    M->nparam = L.total_trained;
    const size_t nw = (size_t)in_dim * hidden1 + (size_t)hidden1 * hidden2 + hidden2;
    bool ok = !alloc_should_fail();
    ok = ok && cudaMalloc(&M->params, sizeof(float) * L.total) == cudaSuccess;
    ok = ok && cudaMalloc(&M->grads, sizeof(float) * L.total_trained) == cudaSuccess;
    ok = ok && cudaMalloc(&M->adam_m, sizeof(float) * L.total_trained) == cudaSuccess;
    ok = ok && cudaMalloc(&M->adam_v, sizeof(float) * L.total_trained) == cudaSuccess;
    ok = ok && cudaMalloc(&M->wbf, sizeof(__nv_bfloat16) * nw) == cudaSuccess;
    ok = ok && cudaMalloc(&M->work, sizeof(float) * work_floats(in_dim, hidden1, hidden2,
                                                                  max_batch)) == cudaSuccess;
    ok = ok && cudaMalloc(&M->loss, sizeof(float)) == cudaSuccess;
    if (ok) {
        ok = cudaMemset(M->params, 0, sizeof(float) * L.total) == cudaSuccess &&
             cudaMemset(M->adam_m, 0, sizeof(float) * L.total_trained) == cudaSuccess &&
             cudaMemset(M->adam_v, 0, sizeof(float) * L.total_trained) == cudaSuccess;
    }
    if (!ok) {
        cudaGetLastError();
        hc_mlp_free(M);
        return HC_ERR_OOM;
    }
    *out = M;
    return HC_OK;
}

HC_API uint32_t hc_mlp_param_count(const hc_mlp* M) { return M ? M->nparam : 0; }

HC_API int hc_mlp_set_params(hc_mlp* M, const float* params_host, const float* mu_host,
                             const float* isd_host) {
    if (!M || !params_host || !mu_host || !isd_host) return HC_ERR_ARG;
    const Layout L = layout_of(M->in, M->h1, M->h2);
    if (cudaMemcpy(M->params, params_host, sizeof(float) * L.total_trained,
                   cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(M->params + L.mu, mu_host, sizeof(float) * M->in, cudaMemcpyHostToDevice) !=
            cudaSuccess ||
        cudaMemcpy(M->params + L.isd, isd_host, sizeof(float) * M->in, cudaMemcpyHostToDevice) !=
            cudaSuccess ||
        cudaMemset(M->adam_m, 0, sizeof(float) * L.total_trained) != cudaSuccess ||
        cudaMemset(M->adam_v, 0, sizeof(float) * L.total_trained) != cudaSuccess)
        return HC_ERR_CUDA;
    M->steps = 0;
    M->bf_stale = true;
    return HC_OK;
}

HC_API int hc_mlp_get_params(const hc_mlp* M, float* params_host, float* mu_host, float* isd_host) {
    if (!M || !params_host) return HC_ERR_ARG;
    const Layout L = layout_of(M->in, M->h1, M->h2);
    if (cudaMemcpy(params_host, M->params, sizeof(float) * L.total_trained,
                   cudaMemcpyDeviceToHost) != cudaSuccess)
        return HC_ERR_CUDA;
    if (mu_host && cudaMemcpy(mu_host, M->params + L.mu, sizeof(float) * M->in,
                              cudaMemcpyDeviceToHost) != cudaSuccess)
        return HC_ERR_CUDA;
    if (isd_host && cudaMemcpy(isd_host, M->params + L.isd, sizeof(float) * M->in,
                               cudaMemcpyDeviceToHost) != cudaSuccess)
        return HC_ERR_CUDA;
    return HC_OK;
}

HC_API int hc_mlp_gradients(hc_mlp* M, const float* x_dev, const float* t_dev, uint32_t n,
                            float* grads_dev, float* loss_host, void* cuda_stream) {
    if (!M || n < 1 || n > M->max_batch || !dev_ptr(x_dev) || !dev_ptr(t_dev)) return HC_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    if (int rc = launch_layers(M, x_dev, t_dev, nullptr, n, nullptr, s)) return rc;
    if (int rc = launch_grads(M, n, nullptr, s)) return rc;
    if (grads_dev && cudaMemcpyAsync(grads_dev, M->grads, sizeof(float) * M->nparam,
                                     cudaMemcpyDeviceToDevice, s) != cudaSuccess)
        return HC_ERR_CUDA;
    return loss_host ? read_loss(M, n, loss_host, s) : HC_OK;
}

}  // extern "C"

namespace {
// forward, backward and one Adam step (beta 0.9 / 0.999, eps 1e-8) on a batch:
// rows perm[0 .. n) of x and t, or the first n when perm is null
int train_step(hc_mlp* M, const float* x_dev, const float* t_dev, const uint32_t* perm, uint32_t n,
               float lr, cudaStream_t s) {
    if (int rc = launch_layers(M, x_dev, t_dev, perm, n, nullptr, s)) return rc;
    M->steps += 1;
    const double b1 = 0.9, b2 = 0.999;
    const float c1 = (float)(1.0 - std::pow(b1, (double)M->steps));
    const float c2 = (float)(1.0 - std::pow(b2, (double)M->steps));
    const Adam adam{lr, (float)b1, (float)b2, 1e-8f, c1, c2};
    M->bf_stale = true;
    return launch_grads(M, n, &adam, s);
}
}  // namespace

extern "C" {

HC_API int hc_mlp_train_step(hc_mlp* M, const float* x_dev, const float* t_dev, uint32_t n,
                             float lr, float* loss_host, void* cuda_stream) {
    if (!M || n < 1 || n > M->max_batch || !(lr > 0.f)) return HC_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    if (int rc = train_step(M, x_dev, t_dev, nullptr, n, lr, s)) return rc;
    return loss_host ? read_loss(M, n, loss_host, s) : HC_OK;
}

HC_API int hc_mlp_fit(hc_mlp* M, const float* feat_dev, const uint32_t* labels_dev, uint32_t n,
                      uint32_t epochs, uint32_t batch, float lr, uint64_t seed, float* losses_host,
                      void* cuda_stream) {
    TraceRange tr("hc_mlp_fit");
    if (!M || batch < 1 || batch > M->max_batch || n < batch || epochs < 1 || !(lr > 0.f) ||
        !losses_host || !dev_ptr(feat_dev) || !dev_ptr(labels_dev))
        return HC_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    const Layout L = layout_of(M->in, M->h1, M->h2);
    const uint32_t nbatch = n / batch;              // whole minibatches per epoch
    const uint32_t every = 50;                      // minibatches between recorded losses
    const uint32_t logs = (nbatch + every - 1) / every;
    // scratch: targets | sort keys | sorted keys (two) | permutation | column sums | losses | sort
    SortProblem sp;
    sp.seg_off = {0, (uint64_t)n};
    sp.key_bits = 32;
    const size_t stats = (size_t)M->in * kStatGroups;
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const size_t o_t = 0, o_keys = al(4ull * n), o_sh = o_keys + al(8ull * n),
                 o_sl = o_sh + al(8ull * n), o_perm = o_sl + al(8ull * n),
                 o_seg = o_perm + al(4ull * n), o_stat = o_seg + 256,
                 o_log = o_stat + al(16 * stats),
                 o_sort = o_log + al(4ull * logs * epochs), bytes = o_sort + sort_scratch_bytes(sp);
    if (alloc_should_fail()) return HC_ERR_OOM;
    char* buf = nullptr;
    if (cudaMallocAsync((void**)&buf, bytes, s) != cudaSuccess) {
        cudaGetLastError();
        return HC_ERR_OOM;
    }
    float* t = reinterpret_cast<float*>(buf + o_t);
    uint64_t* keys = reinterpret_cast<uint64_t*>(buf + o_keys);
    uint32_t* perm = reinterpret_cast<uint32_t*>(buf + o_perm);
    uint64_t* seg = reinterpret_cast<uint64_t*>(buf + o_seg);   // seg_off[2], id_base[1]
    double* sums = reinterpret_cast<double*>(buf + o_stat);
    float* lg = reinterpret_cast<float*>(buf + o_log);
    int rc = HC_OK;
    fit_targets_kernel<<<(n + 255) / 256, 256, 0, s>>>(labels_dev, n, t);
    const dim3 stat_grid(M->in, kStatGroups);
    fit_stats_kernel<false><<<stat_grid, 32, 0, s>>>(feat_dev, n, M->in, sums, sums + stats);
    fit_stats_kernel<true><<<stat_grid, 32, 0, s>>>(feat_dev, n, M->in, sums, sums + stats);
    fit_norm_kernel<<<1, kMaxDim, 0, s>>>(n, M->in, sums, sums + stats, M->params + L.mu,
                                          M->params + L.isd);
    count_launches(4);
    const uint64_t small[3] = {0, (uint64_t)n, 0};
    if (upload_small(seg, small, sizeof(small), s) != cudaSuccess) rc = HC_ERR_CUDA;
    sp.seg_off_dev = seg;
    sp.hi = keys;   // carried along; only the 32 key bits in the low word are compared
    sp.lo = keys;
    sp.ids = nullptr;
    sp.id_base_dev = seg + 2;   // ids = positions: the sorted ids are the permutation
    sp.out_hi = reinterpret_cast<uint64_t*>(buf + o_sh);
    sp.out_lo = reinterpret_cast<uint64_t*>(buf + o_sl);
    sp.out_ids = perm;
    sp.ids_only = true;
    std::vector<float> host_log((size_t)logs * epochs, 0.f);
    for (uint32_t e = 0; !rc && e < epochs; ++e) {
        fit_keys_kernel<<<(n + 255) / 256, 256, 0, s>>>(seed, e, n, keys);
        count_launches(1);
        if (cudaGetLastError() != cudaSuccess || (rc = sort_segments(sp, buf + o_sort, s))) {
            if (!rc) rc = HC_ERR_CUDA;
            break;
        }
        for (uint32_t j = 0; !rc && j < nbatch; ++j) {
            rc = train_step(M, feat_dev, t, perm + (size_t)j * batch, batch, lr, s);
            if (!rc && j % every == 0) rc = launch_loss(M, batch, s);
            if (!rc && j % every == 0 &&
                cudaMemcpyAsync(lg + (size_t)e * logs + j / every, M->loss, sizeof(float),
                                cudaMemcpyDeviceToDevice, s) != cudaSuccess)
                rc = HC_ERR_CUDA;
        }
    }
    if (!rc && (cudaMemcpyAsync(host_log.data(), lg, sizeof(float) * host_log.size(),
                                cudaMemcpyDeviceToHost, s) != cudaSuccess ||
                cudaStreamSynchronize(s) != cudaSuccess))
        rc = HC_ERR_CUDA;
    cudaFreeAsync(buf, s);
    cudaStreamSynchronize(s);
    if (rc) {
        cudaGetLastError();
        return rc;
    }
    for (uint32_t e = 0; e < epochs; ++e) {
        double sum = 0.0;
        for (uint32_t j = 0; j < logs; ++j) sum += host_log[(size_t)e * logs + j];
        losses_host[e] = (float)(sum / logs);
    }
    return HC_OK;
}

HC_API int hc_mlp_forward(hc_mlp* M, const float* x_dev, uint32_t n, int bf16, float* y_dev,
                          void* cuda_stream) {
    if (!M || !dev_ptr(x_dev) || !dev_ptr(y_dev)) return HC_ERR_ARG;
    if (n == 0) return HC_OK;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    if (!bf16) return launch_layers(M, x_dev, nullptr, nullptr, n, y_dev, s);
    if (int rc = refresh_bf16(M, s)) return rc;
    const MlpView V = view_of_mlp(M);
    const size_t smem = pred_smem(V.in, V.h1, V.h2);
    if (allow_shared(mlp_infer_kernel, pred_smem(kMaxDim, kMaxDim, kMaxDim)) != cudaSuccess)
        return HC_ERR_CUDA;
    unsigned blocks = (n + kPredWarps - 1) / kPredWarps;
    if (blocks > 2048) blocks = 2048;
    mlp_infer_kernel<<<blocks, kPredWarps * 32, smem, s>>>(V, x_dev, n, y_dev);
    count_launches(1);
    return cudaGetLastError() == cudaSuccess ? HC_OK : HC_ERR_CUDA;
}

HC_API int hc_mlp_predict_depths(hc_mlp* M, hc_index* idx, const void* q_dev, uint32_t nq,
                                 float margin, uint32_t p_lo, uint32_t p_hi, uint32_t* p_dev,
                                 void* cuda_stream) {
    TraceRange tr("hc_mlp_predict_depths");
    if (!M || features_ok(idx) != HC_OK || M->in != 4 * idx->params.curves) return HC_ERR_ARG;
    if (p_lo > p_hi || p_hi > (1u << 30)) return HC_ERR_ARG;
    if (nq == 0) return HC_OK;
    if (!dev_ptr(q_dev) || !dev_ptr(p_dev) || ((uintptr_t)q_dev & 15)) return HC_ERR_ARG;
    return launch_predict_depths(M, idx, q_dev, nq, margin, p_lo, p_hi, p_dev,
                                 static_cast<cudaStream_t>(cuda_stream)) == cudaSuccess
               ? HC_OK
               : HC_ERR_CUDA;
}

HC_API void hc_mlp_free(hc_mlp* M) {
    if (!M) return;
    cudaFree(M->params);
    cudaFree(M->grads);
    cudaFree(M->adam_m);
    cudaFree(M->adam_v);
    cudaFree(M->wbf);
    cudaFree(M->work);
    cudaFree(M->loss);
    cudaGetLastError();
    delete M;
}

}  // extern "C"
