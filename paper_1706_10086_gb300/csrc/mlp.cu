// Learned tile-config cost model: an FP32 MLP 7 -> 64 -> 64 -> C (ReLU), one
// output per tile config (native configs first, then the emulated path's),
// trained on the autotuner's timings to predict ln(time / best time) of every
// config for an unseen (M, N, K, path).  The paper tunes its tile size by hand
// per architecture (Sect. 3, Table 4); the model generalises that sweep.
//
// Kernels (all hand-written, FP32, fixed summation order, so results are
// deterministic):
//   features   x = (log2 M, log2 N, log2 K, log2 M/N, log2 N/K, log2 M/K, path),
//              standardised with a per-feature mean and standard deviation;
//   forward    z1 = W1 x + b1, h1 = relu(z1), z2 = W2 h1 + b2, h2 = relu(z2),
//              y = W3 h2 + b3 (16 samples per block, weights in shared memory);
//   backward   masked MSE L = sum m (y - t)^2 / sum m: deltas of 16 samples per
//              block with their share of the loss, then the gradients as
//              products over the batch, shared by the blocks of a cluster;
//   adam       elementwise Adam with bias correction (Kingma and Ba 2015).
// All are small (0.23 GFLOP and 6 MB for 4000 samples and 78 outputs), so they
// are bound by latency: what counts is the blocks in flight and the length of
// each serial chain.  One training step of that size on GB300: 1061 -> 43.1 us
// (forward 130 -> 10, loss and deltas 676 -> 12, gradients 432 -> 15, Adam 4).
// Parameters are one float array: W1[64][7], b1[64], W2[64][64], b2[64],
// W3[C][64], b3[C].
#include <atomic>
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "alp_ext.h"
#include "alp_internal.cuh"
#include "tc.cuh"

namespace alp {

std::vector<alp_config> configs_of(alp_path path);

namespace {

constexpr int kF = 7, kH = 64;

__host__ __device__ constexpr int64_t off_w1() { return 0; }
__host__ __device__ constexpr int64_t off_b1() { return kH * kF; }
__host__ __device__ constexpr int64_t off_w2() { return kH * kF + kH; }
__host__ __device__ constexpr int64_t off_b2() { return kH * kF + kH + kH * kH; }
__host__ __device__ constexpr int64_t off_w3() { return kH * kF + 2 * kH + kH * kH; }
__host__ __device__ inline int64_t off_b3(int C) { return off_w3() + (int64_t)C * kH; }
__host__ __device__ inline int64_t param_count(int C) { return off_b3(C) + C; }

__global__ void features_kernel(int64_t n, const int64_t* __restrict__ M,
                                const int64_t* __restrict__ N, const int64_t* __restrict__ K,
                                const int32_t* __restrict__ path, const float* __restrict__ mean,
                                const float* __restrict__ stdv, float* __restrict__ X) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float lm = log2f((float)M[i]), ln = log2f((float)N[i]), lk = log2f((float)K[i]);
    float f[kF] = {lm, ln, lk, lm - ln, ln - lk, lm - lk, (float)path[i]};
#pragma unroll
    for (int j = 0; j < kF; ++j) {
        float v = f[j];
        if (mean) v = (v - mean[j]) / stdv[j];
        X[i * kF + j] = v;
    }
}

// mean and standard deviation (population; 1 where it would be 0) per feature
__global__ void stats_kernel(int64_t n, const float* __restrict__ X, float* mean, float* stdv) {
    const int j = threadIdx.x;
    if (j >= kF) return;
    double s = 0.0, s2 = 0.0;
    for (int64_t i = 0; i < n; ++i) {
        const double v = X[i * kF + j];
        s += v;
        s2 += v * v;
    }
    const double mu = n > 0 ? s / n : 0.0;
    double var = n > 0 ? s2 / n - mu * mu : 0.0;
    if (var < 1e-12) var = 1.0;
    mean[j] = (float)mu;
    stdv[j] = (float)sqrt(var);
}

constexpr int kRows = 16;            // samples per block (forward, deltas)
constexpr int kMlpThreads = 256;     // 64 columns x 4 groups of 4 samples
constexpr int kWPad = kH + 1;        // row stride of a staged 64 x 64 weight tile

// Stages rows row0.. of a row-major (rows x 64) weight matrix, at most 64 of
// them (zeros past the last), into w with row stride LD (kWPad where a warp
// reads a column of it, kH where it reads a row).
template <int LD>
__device__ __forceinline__ void stage_weights(const float* __restrict__ W, int row0, int rows,
                                              float* w) {
    constexpr int kStep = kMlpThreads / kH;   // rows per pass
    const int r = threadIdx.x / kH, left = rows - row0 - r;
    const float* p = W + (int64_t)row0 * kH + threadIdx.x;
    float* o = w + r * LD + threadIdx.x % kH;
#pragma unroll
    for (int i = 0; i < kH / kStep; ++i)
        o[i * kStep * LD] = i * kStep < left ? __ldg(p + i * kMlpThreads) : 0.f;
}

// z[0..3] += sum_k w[j][k] h[k][4 g .. 4 g + 3]
__device__ __forceinline__ void dot4(const float* w, const float (*h)[kRows], int j, int g,
                                     float (&z)[4]) {
#pragma unroll 16
    for (int k = 0; k < kH; ++k) {
        const float x = w[j * kWPad + k];
        const float4 v = *reinterpret_cast<const float4*>(&h[k][4 * g]);
        z[0] = fmaf(x, v.x, z[0]);
        z[1] = fmaf(x, v.y, z[1]);
        z[2] = fmaf(x, v.z, z[2]);
        z[3] = fmaf(x, v.w, z[3]);
    }
}

// 16 samples per block, thread (j, g) the j-th unit of samples 4 g .. 4 g + 3.
// One block per sample read 38 KB of weights from L2 for 10,000 multiply-adds:
// 130 us for 4000 samples and 78 outputs; the staged weights serve 16 samples.
__global__ void __launch_bounds__(kMlpThreads) forward_kernel(const float* __restrict__ P, int C,
                                                              const float* __restrict__ X,
                                                              int64_t B, float* __restrict__ Y,
                                                              float* __restrict__ cache) {
    __shared__ float w2[kH * kWPad], w3[kH * kWPad];
    __shared__ __align__(16) float x[8][kRows], h1[kH][kRows], h2[kH][kRows];
    const int64_t n0 = (int64_t)blockIdx.x * kRows;
    const int j = threadIdx.x & 63, g = threadIdx.x >> 6;
    if (threadIdx.x < kRows * kF) {
        const int r = threadIdx.x / kF, f = threadIdx.x % kF;
        x[f][r] = n0 + r < B ? X[(n0 + r) * kF + f] : 0.f;
    }
    stage_weights<kWPad>(P + off_w2(), 0, kH, w2);
    stage_weights<kWPad>(P + off_w3(), 0, C, w3);
    float w1[kF];
#pragma unroll
    for (int f = 0; f < kF; ++f) w1[f] = P[off_w1() + j * kF + f];
    float z[4];
    const float b1 = P[off_b1() + j], b2 = P[off_b2() + j];
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        z[u] = b1;
#pragma unroll
        for (int f = 0; f < kF; ++f) z[u] = fmaf(w1[f], x[f][4 * g + u], z[u]);
        if (n0 + 4 * g + u < B) cache[(n0 + 4 * g + u) * 2 * kH + j] = z[u];
        h1[j][4 * g + u] = z[u] > 0.f ? z[u] : 0.f;
        z[u] = b2;
    }
    __syncthreads();
    dot4(w2, h1, j, g, z);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        if (n0 + 4 * g + u < B) cache[(n0 + 4 * g + u) * 2 * kH + kH + j] = z[u];
        h2[j][4 * g + u] = z[u] > 0.f ? z[u] : 0.f;
    }
    for (int c0 = 0; c0 < C; c0 += kH) {
        if (c0) {
            __syncthreads();
            stage_weights<kWPad>(P + off_w3(), c0, C, w3);
        }
        __syncthreads();
        const int c = c0 + j;
        if (c >= C) continue;
        const float b3 = P[off_b3(C) + c];
#pragma unroll
        for (int u = 0; u < 4; ++u) z[u] = b3;
        dot4(w3, h2, j, g, z);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (n0 + 4 * g + u < B) Y[(n0 + 4 * g + u) * C + c] = z[u];
    }
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The block's sums of a and b (b held by lane 0 of each warp only), in thread
// 0; red: 2 * kMlpThreads / 32 doubles.  An FP64 addition holds a sub-partition
// for 73 clocks, so only warp 0 adds the warps' sums, both at once in two
// lanes.  Every thread passes its barrier.
__device__ __forceinline__ void block_sums(double& a, double& b, double* red) {
    constexpr int kW = kMlpThreads / 32;
    a = warp_sum(a);
    if ((threadIdx.x & 31) == 0) {
        red[threadIdx.x >> 5] = a;
        red[kW + (threadIdx.x >> 5)] = b;
    }
    __syncthreads();
    if (threadIdx.x >= 32) return;
    const double* r = red + (threadIdx.x & 1) * kW;
    a = r[0];
#pragma unroll
    for (int i = 1; i < kW; ++i) a += r[i];
    b = __shfl_sync(0xffffffffu, a, 1);
}

// The exact double of a float that is zero or normal, by its bits: a
// conversion holds the FP64 unit for as long as an addition does.
__device__ __forceinline__ double widen(float x) {
    const uint32_t u = __float_as_uint(x), e = (u << 1) ? 896u << 20 : 0u;
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + e)),
                            (int)(u << 29));
}
__device__ __forceinline__ bool zero_or_normal(float x) {
    const uint32_t e = (__float_as_uint(x) >> 23) & 255u;
    return e - 1u < 254u || (__float_as_uint(x) << 1) == 0u;
}

// A double as two floats' bits in an array aligned to 4 bytes only.
__device__ __forceinline__ void store_double(float* p, double v) {
    p[0] = __int_as_float(__double2loint(v));
    p[1] = __int_as_float(__double2hiint(v));
}
__device__ __forceinline__ double load_double(const float* p) {
    return __hiloint2double(__float_as_int(p[1]), __float_as_int(p[0]));
}

// Per-sample deltas without the loss's 1 / sum m (grad_kernel applies it):
// dy = 2 m (y - t), dz2 = (W3^T dy) * [z2 > 0], dz1 = (W2^T dz2) * [z1 > 0]
// (dz[n] = dz1, dz2), 16 samples per block as in the forward, and the block's
// sums of m (y - t)^2 and m in double: into part[4 * block] (the bits of
// both doubles), or, from the only block of a launch, finished into lossc.  The
// loss and its count were a kernel of one block, 657 us for 4000 x 78 elements.
__global__ void __launch_bounds__(kMlpThreads) delta_kernel(
    const float* __restrict__ P, int C, int64_t B, const float* __restrict__ cache,
    const float* __restrict__ Y, const float* __restrict__ T, const float* __restrict__ Mk,
    float* __restrict__ part, float* __restrict__ dz, float* __restrict__ lossc) {
    __shared__ __align__(16) float d[kH][kRows];   // a chunk of dy, then dz2, by column
    __shared__ float w3[kH * kH], w2[kH * kH];
    __shared__ double red[2 * kMlpThreads / 32];
    const int64_t n0 = (int64_t)blockIdx.x * kRows;
    const int j = threadIdx.x & 63, g = threadIdx.x >> 6;
    // every load of a chunk in flight before the first use
    float m[4], y[4], t[4], z1[4], z2[4];
    const int64_t at = (n0 + 4 * g) * C + j;
    const int rows = (int)(B - n0 - 4 * g < 4 ? B - n0 - 4 * g : 4);
    auto load = [&](int c0) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t i = at + c0 + (int64_t)u * C;
            const bool in = c0 + j < C && u < rows;
            m[u] = in ? __ldg(Mk + i) : 0.f;
            y[u] = in ? __ldg(Y + i) : 0.f;
            t[u] = in ? __ldg(T + i) : 0.f;
        }
    };
    load(0);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int64_t n = n0 + 4 * g + u;
        z1[u] = n < B ? __ldg(cache + n * 2 * kH + j) : 0.f;
        z2[u] = n < B ? __ldg(cache + n * 2 * kH + kH + j) : 0.f;
    }
    stage_weights<kH>(P + off_w2(), 0, kH, w2);
    // A warp whose mask is zeros and ones and whose values are zero or normal
    // (the tuner's own data) takes two FP64 operations per element, the others
    // seven: the sums are the same, as products with 1 and counts are exact.
    // (At 73 clocks each the seven took the step 48.9 us, the two 44.7.)
    double sum = 0.0, cnt = 0.0;
    int ones = 0;           // elements counted by the first kind
    bool others = false;    // cnt is in use (uniform in a warp)
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    auto dot = [&](const float* w, int rows) {   // v += w^T d over the rows of w
#pragma unroll 16
        for (int k = 0; k < rows; ++k) {
            const float x = w[k * kH + j];
            const float4 e = *reinterpret_cast<const float4*>(&d[k][4 * g]);
            v[0] = fmaf(x, e.x, v[0]);
            v[1] = fmaf(x, e.y, v[1]);
            v[2] = fmaf(x, e.z, v[2]);
            v[3] = fmaf(x, e.w, v[3]);
        }
    };
    for (int c0 = 0; c0 < C; c0 += kH) {
        if (c0) __syncthreads();
        stage_weights<kH>(P + off_w3(), c0, C, w3);
        if (c0 + (j & 32) < C) {   // whole warps past the last column skip the FP64 sums
            bool plain = true;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                plain = plain && (m[u] == 0.f || m[u] == 1.f) && zero_or_normal(y[u]) &&
                        zero_or_normal(t[u]);
            if (__all_sync(0xffffffffu, plain)) {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const bool on = m[u] != 0.f;
                    const double e = widen(on ? y[u] : 0.f) - widen(on ? t[u] : 0.f);
                    sum = fma(e, e, sum);
                    ones += on;
                }
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const double e = (double)y[u] - (double)t[u];
                    sum += m[u] * e * e;
                    cnt += m[u];
                }
                others = true;
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) d[j][4 * g + u] = 2.0f * m[u] * (y[u] - t[u]);
        __syncthreads();
        if (c0 + kH < C) load(c0 + kH);
        dot(w3, C - c0 < kH ? C - c0 : kH);
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int64_t n = n0 + 4 * g + u;
        const float d2 = z2[u] > 0.f ? v[u] : 0.f;
        if (n < B) dz[n * 2 * kH + kH + j] = d2;
        d[j][4 * g + u] = d2;
        v[u] = 0.f;
    }
    ones = __reduce_add_sync(0xffffffffu, ones);
    if (others) cnt = warp_sum(cnt);
    if ((threadIdx.x & 31) == 0) cnt += ones;
    block_sums(sum, cnt, red);   // its barrier also makes d visible
    dot(w2, kH);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int64_t n = n0 + 4 * g + u;
        if (n < B) dz[n * 2 * kH + j] = z1[u] > 0.f ? v[u] : 0.f;
    }
    if (threadIdx.x == 0) {
        if (gridDim.x == 1) {
            lossc[0] = (float)(cnt > 0 ? sum / cnt : 0.0);
            lossc[1] = (float)cnt;
        } else {
            float* o = part + 4 * (int64_t)blockIdx.x;
            store_double(o, sum);
            store_double(o + 2, cnt);
        }
    }
}

// Gradients: eight rows of W3, W2 or W1 (with their biases) per cluster, whose
// eight blocks share the batch: G[r][c] = sum_n D[n][r] H[n][c] / sum m with
// (D, H) = (dy, h2), (dz2, h1), (dz1, x).  64 samples at a time are staged (the
// next 64 loaded before this 64's products); each warp takes every eighth
// sample and two columns per lane.  The warps' partial sums are added in
// shared memory, the blocks' through distributed shared memory, in a fixed
// order.  (One thread per parameter walking the whole batch: 432 us.)
constexpr int kGradRows = 8, kGradChunk = 64, kGradCluster = 8;
constexpr int kGradOut = kGradRows * (kH + 1);   // a tile's gradients, biases last

__global__ void __launch_bounds__(kMlpThreads) grad_kernel(
    const float* __restrict__ X, int C, int64_t B, const float* __restrict__ cache,
    const float* __restrict__ Y, const float* __restrict__ T, const float* __restrict__ Mk,
    const float* __restrict__ part, int nparts, const float* __restrict__ dz,
    float* __restrict__ G, float* __restrict__ lossc) {
    constexpr int kWarps = kMlpThreads / 32;
    __shared__ __align__(16) float sd[kGradChunk][kGradRows];
    __shared__ __align__(16) float sh[kGradChunk][kH];
    __shared__ float sums[kGradOut];
    __shared__ float s_inv;   // 1 / sum m
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t rank = cluster_ctarank();
    const int tile = blockIdx.x / kGradCluster;
    const int t3 = (C + kGradRows - 1) / kGradRows, t2 = kH / kGradRows;
    const int seg = tile < t3 ? 3 : tile < t3 + t2 ? 2 : 1;   // W3, W2 or W1
    const int r0 = (seg == 3 ? tile : seg == 2 ? tile - t3 : tile - t3 - t2) * kGradRows;
    const int64_t lo = B * rank / kGradCluster, hi = B * (rank + 1) / kGradCluster;

    // operand sources of the tile's segment, so that a chunk's loads are plain
    // predicated ones, all in flight together
    const bool w3 = seg == 3;
    const float* dsrc = w3 ? Y + r0 : dz + (seg == 2 ? kH : 0) + r0;
    const float* hsrc = seg == 1 ? X : cache + (w3 ? kH : 0);
    const int64_t dld = w3 ? C : 2 * kH, hld = seg == 1 ? kF : 2 * kH;
    const int dcols = w3 ? min(C - r0, kGradRows) : kGradRows, hcols = seg == 1 ? kF : kH;
    constexpr int kD = kGradChunk * kGradRows / kMlpThreads, kHn = kGradChunk * kH / kMlpThreads;
    constexpr int kDStep = kMlpThreads / kGradRows, kHStep = kMlpThreads / kH;   // samples
    const int dn = tid / kGradRows, dr = tid % kGradRows, hn = tid / kH, hc = tid % kH;
    const bool din = dr < dcols, hin = hc < hcols;
    // this thread's first elements of the next chunk to load, which advance by
    // chunks (with indices formed anew for each load a training step took 44.7
    // us, 43.1 this way)
    const float* dp = dsrc + (lo + dn) * dld + dr;
    const float* tp = T + (lo + dn) * C + r0 + dr;
    const float* mp = Mk + (lo + dn) * C + r0 + dr;
    const float* hp = hsrc + (lo + hn) * hld + hc;
    int left = (int)(hi - lo);   // samples not loaded yet
    float rd[kD], rt[kD], rm[kD], rh[kHn];
    auto load = [&]() {
#pragma unroll
        for (int i = 0; i < kD; ++i) {
            const bool in = din && dn + i * kDStep < left;
            rd[i] = in ? dp[i * kDStep * dld] : 0.f;
            rt[i] = in && w3 ? __ldg(tp + i * kDStep * (int64_t)C) : 0.f;
            rm[i] = in && w3 ? __ldg(mp + i * kDStep * (int64_t)C) : 0.5f;   // 2 m (y - t) = dz below
        }
#pragma unroll
        for (int i = 0; i < kHn; ++i)
            rh[i] = hin && hn + i * kHStep < left ? __ldg(hp + i * kHStep * hld) : 0.f;
        dp += kGradChunk * dld;
        tp += kGradChunk * (int64_t)C;
        mp += kGradChunk * (int64_t)C;
        hp += kGradChunk * hld;
        left -= kGradChunk;
    };
    float acc[kGradRows][2], bias = 0.f;
#pragma unroll
    for (int r = 0; r < kGradRows; ++r) acc[r][0] = acc[r][1] = 0.f;
    if (left > 0) load();
    // while those arrive, one warp adds the delta blocks' mask counts (and, in
    // the first block, their losses): the same sum in every block
    if (warp == kWarps - 1) {
        float count = nparts > 1 ? 0.f : lossc[1];
        if (nparts > 1) {
            double sum = 0.0, cnt = 0.0;
            for (int i = lane; i < nparts; i += 32) {
                cnt += load_double(part + 4 * (int64_t)i + 2);
                if (blockIdx.x == 0) sum += load_double(part + 4 * (int64_t)i);
            }
            cnt = warp_sum(cnt);
            count = (float)cnt;
            if (blockIdx.x == 0) {
                sum = warp_sum(sum);
                if (lane == 0) {
                    lossc[0] = (float)(cnt > 0 ? sum / cnt : 0.0);
                    lossc[1] = count;
                }
            }
        }
        if (lane == 0) s_inv = count > 0.f ? 1.0f / count : 0.f;
    }
    for (int64_t n0 = lo; n0 < hi; n0 += kGradChunk) {
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kD; ++i)
            (&sd[0][0])[tid + i * kMlpThreads] = 2.0f * rm[i] * (rd[i] - rt[i]);
#pragma unroll
        for (int i = 0; i < kHn; ++i)
            (&sh[0][0])[tid + i * kMlpThreads] = seg == 1 || rh[i] > 0.f ? rh[i] : 0.f;
        __syncthreads();
        if (left > 0) load();
#pragma unroll
        for (int s = 0; s < kGradChunk / kWarps; ++s) {
            const int n = warp + s * kWarps;
            const float4 d0 = *reinterpret_cast<const float4*>(&sd[n][0]);
            const float4 d1 = *reinterpret_cast<const float4*>(&sd[n][4]);
            const float2 h = *reinterpret_cast<const float2*>(&sh[n][2 * lane]);
            const float dd[kGradRows] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
#pragma unroll
            for (int r = 0; r < kGradRows; ++r) {
                acc[r][0] = fmaf(dd[r], h.x, acc[r][0]);
                acc[r][1] = fmaf(dd[r], h.y, acc[r][1]);
            }
            if (lane < kGradRows) bias += sd[n][lane];
        }
    }
    // the warps' sums meet in the staging buffer: four warps at a time (16 KB
    // hold 4 x kGradOut floats with room)
    float* buf = &sh[0][0];
    for (int half = 0; half < 2; ++half) {
        __syncthreads();
        if (warp / 4 == half) {
            float* o = buf + (warp & 3) * kGradOut;
#pragma unroll
            for (int r = 0; r < kGradRows; ++r)
                *reinterpret_cast<float2*>(o + r * kH + 2 * lane) = make_float2(acc[r][0], acc[r][1]);
            if (lane < kGradRows) o[kGradRows * kH + lane] = bias;
        }
        __syncthreads();
        for (int e = tid; e < kGradOut; e += kMlpThreads) {
            const float v = (buf[e] + buf[kGradOut + e]) + (buf[2 * kGradOut + e] + buf[3 * kGradOut + e]);
            sums[e] = half ? sums[e] + v : v;
        }
    }
    cluster_sync_all();
    const float inv = s_inv;
    for (int e = (int)rank * kMlpThreads + tid; e < kGradOut; e += kGradCluster * kMlpThreads) {
        float s = 0.f;
#pragma unroll
        for (uint32_t q = 0; q < kGradCluster; ++q) {
            float v;
            asm volatile("ld.shared::cluster.f32 %0, [%1];"
                         : "=f"(v)
                         : "r"(cluster_addr(&sums[e], q))
                         : "memory");
            s += v;
        }
        s *= inv;
        const bool is_bias = e >= kGradRows * kH;
        const int r = r0 + (is_bias ? e - kGradRows * kH : e / kH), c = e % kH;
        if (seg == 3) {
            if (r < C) G[is_bias ? off_b3(C) + r : off_w3() + (int64_t)r * kH + c] = s;
        } else if (seg == 2) {
            G[is_bias ? off_b2() + r : off_w2() + r * kH + c] = s;
        } else if (is_bias) {
            G[off_b1() + r] = s;
        } else if (c < kF) {
            G[off_w1() + r * kF + c] = s;
        }
    }
    cluster_sync_all();   // no block leaves while another reads its sums
}

__global__ void adam_kernel(float* __restrict__ P, const float* __restrict__ G,
                            float* __restrict__ m, float* __restrict__ v, int64_t n, float lr,
                            float b1, float b2, float eps, float c1, float c2) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float g = G[i];
    const float mi = b1 * m[i] + (1.f - b1) * g;
    const float vi = b2 * v[i] + (1.f - b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    P[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// ---- the model consulted by alp_tune(PREDICT) and by cfg == NULL calls ----
struct Model {
    bool loaded = false;
    int C = 0;
    std::vector<float> params;
    float mean[kF], stdv[kF];
    int dev = -1;
    float* d_params = nullptr;
    float* d_scratch = nullptr;   // X (7) + Y (C) + cache (128)
    int64_t* d_shape = nullptr;   // M, N, K, path
};
std::mutex g_mmu;
Model g_model;
std::atomic<bool> g_loaded{false};   // g_model.loaded, read without the lock

}  // namespace

bool model_loaded() { return g_loaded.load(); }

// Arg-min of the model's predicted log-time over the valid configs of `path`.
bool model_predict(int64_t M, int64_t N, int64_t K, alp_path path, alp_config* out,
                   double* pred_tflops) {
    std::lock_guard<std::mutex> lk(g_mmu);
    if (!g_model.loaded || M <= 0 || N <= 0 || K <= 0) return false;
    const std::vector<alp_config> nat = configs_of(ALP_PATH_NATIVE);
    const std::vector<alp_config> emu = configs_of(ALP_PATH_EMUL);
    if (g_model.C != (int)(nat.size() + emu.size())) return false;
    int dev = 0;
    cudaGetDevice(&dev);
    const int C = g_model.C;
    if (g_model.dev != dev || !g_model.d_params) {
        if (g_model.d_params) cudaFree(g_model.d_params);
        if (g_model.d_scratch) cudaFree(g_model.d_scratch);
        if (g_model.d_shape) cudaFree(g_model.d_shape);
        g_model.d_params = g_model.d_scratch = nullptr;
        g_model.d_shape = nullptr;
        // one-time upload of the model to this device
        if (cudaMalloc(&g_model.d_params, param_count(C) * 4) != cudaSuccess ||
            cudaMalloc(&g_model.d_scratch, (kF + C + 2 * kH + 2 * kF) * 4) != cudaSuccess ||
            cudaMalloc(&g_model.d_shape, 4 * 8) != cudaSuccess)
            return false;
        float ms[2 * kF];
        std::memcpy(ms, g_model.mean, sizeof g_model.mean);
        std::memcpy(ms + kF, g_model.stdv, sizeof g_model.stdv);
        // scratch layout: X (7) | Y (C) | cache (128) | mean, std (14)
        if (cudaMemcpy(g_model.d_params, g_model.params.data(), param_count(C) * 4,
                       cudaMemcpyHostToDevice) != cudaSuccess ||
            cudaMemcpy(g_model.d_scratch + kF + C + 2 * kH, ms, sizeof ms,
                       cudaMemcpyHostToDevice) != cudaSuccess)
            return false;
        g_model.dev = dev;
    }
    float* X = g_model.d_scratch;
    float* Y = X + kF;
    float* cache = Y + C;
    float* ms = cache + 2 * kH;
    const int64_t h_shape[4] = {M, N, K, path == ALP_PATH_EMUL ? 1 : 0};
    const int32_t h_path = (int32_t)h_shape[3];
    if (cudaMemcpy(g_model.d_shape, h_shape, sizeof h_shape, cudaMemcpyHostToDevice) != cudaSuccess)
        return false;
    if (cudaMemcpy(reinterpret_cast<char*>(g_model.d_shape) + 24, &h_path, 4,
                   cudaMemcpyHostToDevice) != cudaSuccess)
        return false;
    features_kernel<<<1, 32>>>(1, g_model.d_shape, g_model.d_shape + 1, g_model.d_shape + 2,
                               reinterpret_cast<int32_t*>(g_model.d_shape + 3), ms, ms + kF, X);
    forward_kernel<<<1, kMlpThreads>>>(g_model.d_params, C, X, 1, Y, cache);
    std::vector<float> y(C);
    if (cudaMemcpy(y.data(), Y, C * 4, cudaMemcpyDeviceToHost) != cudaSuccess) return false;
    const int lo = path == ALP_PATH_NATIVE ? 0 : (int)nat.size();
    const int hi = path == ALP_PATH_NATIVE ? (int)nat.size() : C;
    int best = lo;
    for (int c = lo; c < hi; ++c)
        if (y[c] < y[best]) best = c;
    *out = path == ALP_PATH_NATIVE ? nat[best] : emu[best - lo];
    if (pred_tflops) *pred_tflops = (double)y[best];   // predicted ln(time / best time)
    return true;
}

}  // namespace alp

using namespace alp;

extern "C" {

int64_t alp_mlp_param_count(int C) { return C > 0 ? param_count(C) : -1; }

alp_status alp_mlp_features(int64_t count, const int64_t* dM, const int64_t* dN,
                            const int64_t* dK, const int32_t* dpath, const float* mean,
                            const float* stdv, float* X, void* stream) {
    if (count < 0 || (count > 0 && (!dM || !dN || !dK || !dpath || !X)) || (!mean != !stdv))
        return ALP_ERR_INVALID_ARG;
    if (count == 0) return ALP_OK;
    features_kernel<<<(unsigned)((count + 255) / 256), 256, 0,
                      reinterpret_cast<cudaStream_t>(stream)>>>(count, dM, dN, dK, dpath, mean,
                                                                stdv, X);
    return cuda_status(cudaGetLastError());
}

alp_status alp_mlp_feature_stats(int64_t count, const float* X, float* mean, float* stdv,
                                 void* stream) {
    if (count < 0 || !X || !mean || !stdv) return ALP_ERR_INVALID_ARG;
    stats_kernel<<<1, 32, 0, reinterpret_cast<cudaStream_t>(stream)>>>(count, X, mean, stdv);
    return cuda_status(cudaGetLastError());
}

alp_status alp_mlp_forward(const float* params, int C, const float* X, int64_t B, float* Y,
                           float* cache, void* stream) {
    if (C <= 0 || B < 0 || B > 0x7fffffff || !params || (B > 0 && (!X || !Y || !cache)))
        return ALP_ERR_INVALID_ARG;
    if (B == 0) return ALP_OK;
    forward_kernel<<<(unsigned)((B + kRows - 1) / kRows), kMlpThreads, 0,
                     reinterpret_cast<cudaStream_t>(stream)>>>(params, C, X, B, Y, cache);
    return cuda_status(cudaGetLastError());
}

alp_status alp_mlp_backward(const float* params, int C, const float* X, int64_t B,
                            const float* cache, const float* Y, const float* T, const float* Mask,
                            float* grads, float* work, float* loss_out, void* stream) {
    if (C <= 0 || B <= 0 || B > 0x7fffffff || !params || !X || !cache || !Y || !T || !Mask ||
        !grads || !work || !loss_out)
        return ALP_ERR_INVALID_ARG;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    // work: the delta blocks' loss parts (4 floats per 16 samples; more than
    // one block has at least 17 samples, so they fit B * C floats), then dz
    float* part = work;
    float* dz = work + B * C;
    const int64_t blocks = (B + kRows - 1) / kRows;
    delta_kernel<<<(unsigned)blocks, kMlpThreads, 0, st>>>(params, C, B, cache, Y, T, Mask, part,
                                                           dz, loss_out);
    const int64_t tiles = (C + kGradRows - 1) / kGradRows + 2 * (kH / kGradRows);
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)(tiles * kGradCluster));
    lc.blockDim = dim3(kMlpThreads);
    lc.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kGradCluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&lc, grad_kernel, X, C, B, cache, Y, T, Mask,
                                             (const float*)part, (int)blocks, (const float*)dz,
                                             grads, loss_out);
    if (e != cudaSuccess) return cuda_status(e);
    return cuda_status(cudaGetLastError());
}

alp_status alp_mlp_adam(float* params, const float* grads, float* m, float* v, int64_t n,
                        int step, float lr, float beta1, float beta2, float eps, void* stream) {
    if (n < 0 || step < 1 || !params || !grads || !m || !v) return ALP_ERR_INVALID_ARG;
    if (n == 0) return ALP_OK;
    const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
    adam_kernel<<<(unsigned)((n + 255) / 256), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
        params, grads, m, v, n, lr, beta1, beta2, eps, c1, c2);
    return cuda_status(cudaGetLastError());
}

alp_status alp_tune_load_model(const float* host_params, int C, const float* host_mean,
                               const float* host_std) {
    if (!host_params || !host_mean || !host_std || C <= 0) return ALP_ERR_INVALID_ARG;
    const int want = (int)(configs_of(ALP_PATH_NATIVE).size() + configs_of(ALP_PATH_EMUL).size());
    if (C != want) return ALP_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lk(g_mmu);
    g_model.params.assign(host_params, host_params + param_count(C));
    std::memcpy(g_model.mean, host_mean, sizeof g_model.mean);
    std::memcpy(g_model.stdv, host_std, sizeof g_model.stdv);
    g_model.C = C;
    g_model.loaded = true;
    g_loaded.store(true);
    g_model.dev = -1;    // re-upload on next use
    return ALP_OK;
}

alp_status alp_tune_unload_model(void) {
    std::lock_guard<std::mutex> lk(g_mmu);
    g_model.loaded = false;
    g_loaded.store(false);
    return ALP_OK;
}

}  // extern "C"
