// Automatic modulus count of the modular emulated GEMM (nslices = 0 with
// ALP_SLICE_BF16_CRT).  The scheme's only error is the rounding of the scaled
// operands A'_ik = RN(A_ik 2^(k - e_i)) and B'_kj = RN(B_kj 2^(k - f_j)), so
// more moduli (a larger k) make it more accurate and slower.  The count is
// chosen from statistics of the operands' rows and columns, read once by the
// kernels below, with an error model of the scheme and one of the native
// FP64 kernel (both stated at crt_moduli_rule); the choice is a heuristic,
// not a bound.
//
// Statistics, with x = |a| 2^-e for the row's (column's) scale exponent e:
//   S1 = sum |x|, S2 = sum x^2 per row of op(A) and per column of op(B);
//   st[0] = max 1/S1^2, st[1] = max S2/S1^2, st[2] = max 1/S2 over the rows
//   of op(A) (all-zero rows skipped), st[3..5] the same over the columns of
//   op(B).  Accumulated in float (a model input; order does not matter).
#include <cmath>

#include "alp_ext.h"
#include "emul.cuh"
#include "emul_prep.cuh"

namespace alp {

namespace {

// |a| 2^-e as a float, for |a| < 2^e: exponent and the top 23 mantissa bits
// of the double; 0 for zeros, subnormals, Inf/NaN (the scan reports those) and
// values below float's normal range (negligible in the sums).
__device__ __forceinline__ float scaled_abs_f32(uint64_t bits, int e) {
    const int ex = (int)((bits >> 52) & 0x7FF);
    if (ex == 0 || ex == 0x7FF) return 0.0f;
    const int fe = ex - 1023 - e + 127;
    if (fe <= 0 || fe >= 255) return 0.0f;
    return __int_as_float((fe << 23) | (int)((bits >> 29) & 0x7FFFFF));
}

// Positive floats order like their bit patterns, so an integer max is a float max.
__device__ __forceinline__ void atomic_max_pos(float* p, float v) {
    atomicMax(reinterpret_cast<int*>(p), __float_as_int(v));
}

// The three statistics of a line, or the largest of several lines'.
struct LineStats {
    float v[3] = {0.0f, 0.0f, 0.0f};
    __device__ __forceinline__ void add(float s1, float s2) {
        if (s1 > 0.0f && s2 > 0.0f) {
            v[0] = fmaxf(v[0], 1.0f / (s1 * s1));
            v[1] = fmaxf(v[1], s2 / (s1 * s1));
            v[2] = fmaxf(v[2], 1.0f / s2);
        }
    }
};

__device__ __forceinline__ void record_stats(const LineStats& s, float* out) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
        if (s.v[i] > 0.0f) atomic_max_pos(out + i, s.v[i]);
}

// The largest of the block's threads' statistics into out, one atomic for
// each: those of every line, all to the same words, queue up in L2 (256^3 with
// the automatic count: 41.7 -> 41.0 us).  All threads call it.
__device__ __forceinline__ void record_block_stats(const LineStats& s, float* out,
                                                   float (*red)[3]) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int m = __reduce_max_sync(0xffffffffu, __float_as_int(s.v[i]));
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][i] = __int_as_float(m);
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        float m = red[0][threadIdx.x];
#pragma unroll
        for (int w = 1; w < kPrepWarps; ++w) m = fmaxf(m, red[w][threadIdx.x]);
        if (m > 0.0f) atomic_max_pos(out + threadIdx.x, m);
    }
}

// Columns of a row-major K x N matrix: blocks of 32 columns x 256 rows, 8
// rows in flight per column; partial sums added into s1[N], s2[N].
constexpr int kStatChunk = 256;
__global__ void crt_stats_cols_kernel(const double* __restrict__ X, int64_t K, int64_t N,
                                      int64_t ldx, const int32_t* __restrict__ f,
                                      float* __restrict__ s1, float* __restrict__ s2) {
    __shared__ float r1[8][33], r2[8][33];
    const int64_t j = (int64_t)blockIdx.x * 32 + threadIdx.x;
    const int64_t k0 = (int64_t)blockIdx.y * kStatChunk;
    const int64_t k1 = (k0 + kStatChunk < K) ? k0 + kStatChunk : K;
    float a1 = 0.0f, a2 = 0.0f;
    if (j < N) {
        const int fj = f[j];
        for (int64_t k = k0 + threadIdx.y; k < k1; k += 8) {
            const float x = scaled_abs_f32((uint64_t)__double_as_longlong(__ldg(X + k * ldx + j)), fj);
            a1 += x;
            a2 = fmaf(x, x, a2);
        }
    }
    r1[threadIdx.y][threadIdx.x] = a1;
    r2[threadIdx.y][threadIdx.x] = a2;
    __syncthreads();
    if (threadIdx.y == 0 && j < N) {
        float t1 = 0.0f, t2 = 0.0f;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            t1 += r1[r][threadIdx.x];
            t2 += r2[r][threadIdx.x];
        }
        atomicAdd(s1 + j, t1);
        atomicAdd(s2 + j, t2);
    }
}

__global__ void crt_stats_finish_kernel(int64_t N, const float* __restrict__ s1,
                                        const float* __restrict__ s2, float* out) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= N) return;
    LineStats s;
    s.add(s1[j], s2[j]);
    record_stats(s, out);
}

// Statistics of the R columns of a row-major L x R matrix X, scale exponents
// `exps`, into out[0..2]; s1, s2: R floats of scratch.
alp_status column_stats(const double* X, int64_t R, int64_t L, int64_t ldx, const int32_t* exps,
                        float* out, float* s1, float* s2, cudaStream_t st) {
    if (R == 0 || L == 0) return ALP_OK;
    if (cudaMemsetAsync(s1, 0, (size_t)R * 4, st) != cudaSuccess ||
        cudaMemsetAsync(s2, 0, (size_t)R * 4, st) != cudaSuccess)
        return ALP_ERR_CUDA;
    const dim3 grid((unsigned)((R + 31) / 32), (unsigned)((L + kStatChunk - 1) / kStatChunk));
    crt_stats_cols_kernel<<<grid, dim3(32, 8), 0, st>>>(X, L, R, ldx, exps, s1, s2);
    crt_stats_finish_kernel<<<(unsigned)((R + 255) / 256), 256, 0, st>>>(R, s1, s2, out);
    return cuda_status(cudaGetLastError());
}

// ---- exponents and statistics of both operands in one launch, with the
// line walks of emul_prep.cuh (contiguous lines by warps or blocks, strided
// ones in strips through shared memory) ----

// The sums of a contiguous line's elements k = 4 t, 4 t + 1, .. of one thread.
template <int TEAM>
__device__ __forceinline__ void stat_line(const double* x, int64_t K, bool vec, int t, int e,
                                          float& s1, float& s2) {
#pragma unroll 1
    for (int64_t k0 = 4 * (int64_t)t; k0 < K; k0 += 16 * TEAM) {
        double a[4][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) prep_load4(x, k0 + (int64_t)q * 4 * TEAM, K, vec, a[q]);
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float v = scaled_abs_f32((uint64_t)__double_as_longlong(a[q][u]), e);
                s1 += v;
                s2 = fmaf(v, v, s2);
            }
    }
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <int TEAM>
__device__ __forceinline__ void stat_rows(const PrepParams<double>& p,
                                          const PrepOperand<double>& o, int block,
                                          LineStats& best, uint64_t (*red)[kPrepWarps],
                                          float2 (*sums)[kPrepWarps]) {
    constexpr int kTeams = kPrepThreads / TEAM;
    const int t = threadIdx.x % TEAM;
    int par = 0;
    for (int64_t r = (int64_t)block * kTeams + threadIdx.x / TEAM; r < o.R;
         r += (int64_t)o.blocks * kTeams, par ^= 1) {
        const double* x = o.X + r * o.ldx;
        const bool vec = (reinterpret_cast<uintptr_t>(x) & 15) == 0;
        const uint64_t mx = prep_line_max<TEAM>(x, p.K, vec, t, red, par);
        const int e = frexp_exponent_of_bits(mx);
        if (t == 0) {
            o.exps[r] = e;
            if (mx >= ScanKey<double>::kInf) set_device_error(p.err, ALP_ERR_UNSUPPORTED);
        }
        float s1 = 0.0f, s2 = 0.0f;
        stat_line<TEAM>(x, p.K, vec, t, e, s1, s2);
        s1 = warp_sum(s1);
        s2 = warp_sum(s2);
        if constexpr (TEAM > 32) {
            if ((t & 31) == 0) sums[par][t >> 5] = make_float2(s1, s2);
            __syncthreads();
            s1 = s2 = 0.0f;
#pragma unroll
            for (int w = 0; w < TEAM / 32; ++w) {
                s1 += sums[par][w].x;
                s2 += sums[par][w].y;
            }
        }
        if (t == 0) best.add(s1, s2);
    }
}

__device__ __forceinline__ void stat_cols(const PrepParams<double>& p,
                                          const PrepOperand<double>& o, int block, double* tile,
                                          LineStats& best, uint64_t* red, uint64_t* cmax,
                                          int* sexp, float2* csum) {
    constexpr int W = kPrepStrip<double>;
    const uint32_t rank = cluster_ctarank(), size = cluster_nctarank();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t j0 = (int64_t)(block / (int)size) * W, kb0 = (int64_t)rank * p.block_k;
    const int rows = (int)min((int64_t)p.block_k, max(p.kpad - kb0, (int64_t)0));
    uint64_t mx[kPrepV<double>];
    prep_fill(o, p.K, j0, kb0, rows, p.block_k, tile, mx);
    const uint64_t m = prep_column_max<double>(mx, red, cmax, size);
    if (threadIdx.x < W) {
        const int e = frexp_exponent_of_bits(m);
        sexp[threadIdx.x] = e;
        if (rank == 0 && j0 + threadIdx.x < o.R) {
            o.exps[j0 + threadIdx.x] = e;
            if (m >= ScanKey<double>::kInf) set_device_error(p.err, ALP_ERR_UNSUPPORTED);
        }
    }
    __syncthreads();
    const int Q = prep_q<double>(p.block_k);
    const double* col = tile + (warp % W) * prep_ld<double>(p.block_k);
    float s1 = 0.0f, s2 = 0.0f;
    for (int k = lane; k < (warp < W ? rows : 0); k += 32) {
        const float v = scaled_abs_f32(
            (uint64_t)__double_as_longlong(col[(k & 3) * Q + (k >> 2)]), sexp[warp % W]);
        s1 += v;
        s2 = fmaf(v, v, s2);
    }
    s1 = warp_sum(s1);
    s2 = warp_sum(s2);
    if (lane == 0 && warp < W) csum[warp] = make_float2(s1, s2);
    cluster_sync_all();
    if (rank == 0 && threadIdx.x < W && j0 + threadIdx.x < o.R) {
        s1 = s2 = 0.0f;
        for (uint32_t q = 0; q < size; ++q) {
            float a, b;
            asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];"
                         : "=f"(a), "=f"(b)
                         : "r"(cluster_addr(&csum[threadIdx.x], q))
                         : "memory");
            s1 += a;
            s2 += b;
        }
        best.add(s1, s2);
    }
    cluster_sync_all();   // csum and cmax read by the whole cluster
}

__global__ void __launch_bounds__(kPrepThreads, 3)
    crt_prep_stats_kernel(const __grid_constant__ PrepParams<double> p, float* out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint64_t red[kPrepWarps * kPrepStrip<double>];
    __shared__ uint64_t cmax[kPrepStrip<double>];
    __shared__ int sexp[kPrepStrip<double>];
    __shared__ __align__(8) float2 sums[2][kPrepWarps];
    const bool second = (int)blockIdx.x >= p.op[0].blocks;
    const PrepOperand<double>& o = p.op[second ? 1 : 0];
    const int block = (int)blockIdx.x - (second ? p.op[0].blocks : 0);
    __shared__ float stats[kPrepWarps][3];
    LineStats best;
    if (o.cols)
        stat_cols(p, o, block, reinterpret_cast<double*>(smem_raw), best, red, cmax, sexp, sums[0]);
    else if (p.K <= kPrepWarpRowK)
        stat_rows<32>(p, o, block, best, reinterpret_cast<uint64_t(*)[kPrepWarps]>(red), sums);
    else
        stat_rows<kPrepThreads>(p, o, block, best,
                                reinterpret_cast<uint64_t(*)[kPrepWarps]>(red), sums);
    record_block_stats(best, out + (second ? 3 : 0), stats);
}

}  // namespace

// The rule.  With u = 2^-53, k = crt_bits(K, n) and the statistics st[6]:
//
//  * the scheme's rounding errors, uniform in half a unit of the scaled
//    operands, give C_ij an error of standard deviation
//    sigma_ij = 2^-k / sqrt(12) * sqrt(4^e_i ||b_j||^2 + 4^f_j ||a_i||^2),
//    and (|A||B|)_ij is about ||a_i||_1 ||b_j||_1 / K, so the largest
//    componentwise error over the M N elements, g = sqrt(2 ln(M N)) standard
//    deviations, is predicted as
//      comp = g / sqrt(12) * 2^(53-k) * K * sqrt(st0 st4 + st3 st1)   [units of u];
//  * the native FP64 kernel's largest componentwise error for operands of
//    one magnitude grows like sqrt(K): modelled as 0.045 sqrt(K) u (4.07 u
//    measured at K = 8192 with this library's DMMA kernel);
//  * normwise, the ratio of the scheme's error to the native kernel's, with
//    the native error modelled as 0.311 u sqrt(K) sqrt(S2_i T2_j / K) per
//    element (calibrated on the same measurement), is
//      norm = 2^(53-k) / (sqrt(12) * 0.311) * sqrt(st2 + st5).
//
// The count is the smallest n with comp <= 0.5 * 0.045 sqrt(K) and norm <=
// 0.5 (half the native kernel's modelled errors, a factor of two against the
// models' own error), else 16.  Operands with an all-zero side give the
// smallest count (the product is exactly zero).
int crt_moduli_rule(int64_t M, int64_t N, int64_t K, const double st[6], double* comp_u,
                    double* norm_ratio) {
    const double kSqrt12 = 3.4641016151377544;
    const double g = std::sqrt(2.0 * std::log((double)(M * N > 2 ? M * N : 2)));
    const double native_comp = 0.045 * std::sqrt((double)(K > 1 ? K : 1));
    const bool zero = !(st[0] > 0.0) || !(st[3] > 0.0);
    int best = 0;
    double c = 0.0, r = 0.0;
    for (int n = kCrtMinModuli; n <= kCrtMaxModuli; ++n) {
        const int k = crt_bits(K, n);
        if (k < 1) continue;
        const double scale = std::ldexp(1.0, 53 - k);
        c = zero ? 0.0 : g / kSqrt12 * scale * (double)K * std::sqrt(st[0] * st[4] + st[3] * st[1]);
        r = zero ? 0.0 : scale / (kSqrt12 * 0.311) * std::sqrt(st[2] + st[5]);
        best = n;
        if (c <= 0.5 * native_comp && r <= 0.5) break;
    }
    if (comp_u) *comp_u = c;
    if (norm_ratio) *norm_ratio = r;
    return best;
}

// Finds the exponents e, f and the statistics of op(A) and op(B) on `stream`,
// waits for them, and applies the rule.  scratch: 8 + 2 max(M, N) floats of
// device memory.
alp_status crt_choose_moduli(int ta, int tb, int64_t M, int64_t N, int64_t K, const double* A,
                             int64_t lda, const double* B, int64_t ldb, int32_t* e, int32_t* f,
                             void* scratch, cudaStream_t stream, int* n_out, double* comp_u,
                             double* norm_ratio) {
    float* out = static_cast<float*>(scratch);
    if (cudaMemsetAsync(out, 0, 8 * sizeof(float), stream) != cudaSuccess) return ALP_ERR_CUDA;
    alp_status st;
    // rows of op(A): rows of A, or columns of its K x M storage; columns of
    // op(B): columns of B, or rows of its N x K storage
    PrepParams<double> p = {};
    p.K = K;
    p.kpad = (K + kEmulBK - 1) / kEmulBK * kEmulBK;
    p.err = device_error_word();
    float* s1 = out + 8;
    float* s2 = s1 + (M > N ? M : N);
    const struct {
        const double* X;
        int64_t R, ldx;
        int cols;
        int32_t* exps;
    } ops[2] = {{A, M, lda, ta, e}, {B, N, ldb, 1 - tb, f}};
    for (int i = 0; i < 2; ++i) {
        const auto& o = ops[i];
        if (!o.cols || prep_in_strips<double>(o.R, K, true))
            p.op[i] = {o.X, o.R, o.ldx, o.exps, nullptr, o.cols, 0};
        else if ((st = emul_exponents<double>(o.R, K, o.X, o.ldx, 1, o.exps, stream)) != ALP_OK ||
                 (st = column_stats(o.X, o.R, K, o.ldx, o.exps, out + 3 * i, s1, s2, stream)) !=
                     ALP_OK)
            return st;
    }
    if ((p.op[0].X || p.op[1].X) &&
        (st = launch_prep_kernel(crt_prep_stats_kernel, p, stream, out)) != ALP_OK)
        return st;
    float h[8];
    if (cudaMemcpyAsync(h, out, sizeof(h), cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
        cudaStreamSynchronize(stream) != cudaSuccess)
        return ALP_ERR_CUDA;
    double sd[6];
    for (int i = 0; i < 6; ++i) sd[i] = h[i];
    const int n = crt_moduli_rule(M, N, K, sd, comp_u, norm_ratio);
    if (n < kCrtMinModuli) return ALP_ERR_UNSUPPORTED;
    *n_out = n;
    return ALP_OK;
}

}  // namespace alp

using namespace alp;

extern "C" {

int alp_emul_crt_moduli_rule(int64_t M, int64_t N, int64_t K, const double* stats,
                             double* predicted) {
    if (M < 0 || N < 0 || K < 0 || K > kCrtMaxK || !stats) return 0;
    double c = 0.0, r = 0.0;
    const int n = crt_moduli_rule(M, N, K, stats, &c, &r);
    if (predicted) {
        predicted[0] = c;
        predicted[1] = r;
    }
    return n;
}

}  // extern "C"
