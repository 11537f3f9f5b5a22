// Native FP64 GEMM without a given tile config: C = alpha op(A) op(B) + beta C
// from register-direct DMMA fragments (native_direct.cuh), the work cut so that
// the 608 sub-partitions finish together.  One 16 x 8 fragment per warp keeps
// the unit of work small; transposed operands are read where they are.
//
// Measured on GB300 through alp_gemm_f64 (us; the shared-memory kernel's
// default config before, this file after; floor 2MNK / 1.098 TFLOP/s):
//   64^3      151.6 ->   6.2          512^3    1168 ->   262 (floor 244)
//   2048^3    18575 -> 15694 (15646)  1021 x 771 x 1333, A^T: 3154 -> 1960 (1911)
// 8192 x 8192 x 2048 runs 249,700 (250,340).  The 64^3 call is bound by its issue;
// its kernel takes 4.7.
#include <algorithm>

#include "alp_ext.h"
#include "native_direct.cuh"
#include "tc.cuh"

namespace alp {

namespace {

constexpr int kWarps = 4;   // one per sub-partition
constexpr int kGroup = 8;   // tile-rows per raster group, for reuse of B's columns in L2

struct DirectParams {
    DirectOperand A, B;
    double* C;
    int64_t ldc, M, N, K;
    double alpha, beta;
    int64_t tiles_m, tiles_n;
    int vec2;   // C and ldc allow 16-byte accesses at even columns
};

__device__ __forceinline__ void tile_of(const DirectParams& p, int64_t tile, int64_t& tm,
                                        int64_t& tn) {
    const int64_t in_group = kGroup * p.tiles_n;
    const int64_t first = tile / in_group * kGroup;
    const int64_t gsz = min(p.tiles_m - first, (int64_t)kGroup);
    const int64_t local = tile % in_group;
    tm = first + local % gsz;
    tn = local / gsz;
}

// A 32 x 16 tile of C per block, 2 x 2 warps.  Bound by the DMMA rate once the
// tiles fill the SMs several times over: 0.998 of it at 2048^3 (0.925 before,
// in waves of 64 x 128 tiles).
__global__ void __launch_bounds__(32 * kWarps) dgemm_direct_kernel(DirectParams p) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int64_t tm, tn;
    tile_of(p, blockIdx.x, tm, tn);
    const int64_t r0 = 32 * tm + 16 * (warp >> 1), c0 = 16 * tn + 8 * (warp & 1);
    Acc<2, 2> acc;
    acc.zero();
    mma_direct<1, 1>(p.A, p.B, p.M, p.N, p.K, r0, c0, 0, (p.K + 3) >> 2, lane, acc);
    epilogue<2, 2>(acc, p.C, p.ldc, p.M, p.N, r0, c0, p.alpha, p.beta, p.vec2 != 0, lane);
}

__device__ __forceinline__ double2 ld_cluster_f64x2(uint32_t addr) {
    double2 v;
    asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];"
                 : "=d"(v.x), "=d"(v.y)
                 : "r"(addr)
                 : "memory");
    return v;
}

// One 16 x 8 fragment of C per cluster of `size` blocks: its k range is cut
// into 4 size parts, one per warp (part 4 rank + warp), so that all four
// sub-partitions of an SM work on it evenly and a shape with few tiles still
// reaches 4 size times as many.  The partial fragments meet in (distributed)
// shared memory and are summed in part order by warps 0 and 1 of the first
// block (one row half each): the order is fixed, so results do not depend on
// timing, and no workspace is needed.
__global__ void __launch_bounds__(32 * kWarps) dgemm_direct_split_kernel(DirectParams p) {
    __shared__ double2 part[kWarps][2][32];   // [warp][row half][lane]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank(), size = cluster_nctarank();
    int64_t tm, tn;
    tile_of(p, blockIdx.x / size, tm, tn);
    const int64_t steps = (p.K + 3) >> 2, parts = kWarps * (int64_t)size;
    const int64_t me = kWarps * (int64_t)rank + warp;
    Acc<2, 2> acc;
    acc.zero();
    mma_direct<1, 1>(p.A, p.B, p.M, p.N, p.K, 16 * tm, 8 * tn, steps * me / parts,
                     steps * (me + 1) / parts, lane, acc);
#pragma unroll
    for (int h = 0; h < 2; ++h)
        part[warp][h][lane] = make_double2(acc.c[0][0][2 * h], acc.c[0][0][2 * h + 1]);
    cluster_sync_all();
    const int64_t r = 16 * tm + 8 * warp + (lane >> 2), c = 8 * tn + 2 * (lane & 3);
    if (rank == 0 && warp < 2 && r < p.M && c < p.N) {
        double s0 = 0.0, s1 = 0.0;
        for (uint32_t q = 0; q < size; ++q) {
            const uint32_t base = cluster_addr(&part[0][warp][lane], q);
#pragma unroll
            for (int w = 0; w < kWarps; ++w) {
                const double2 v = ld_cluster_f64x2(base + (uint32_t)(w * sizeof(part[0])));
                s0 += v.x;
                s1 += v.y;
            }
        }
        double* out = p.C + r * p.ldc + c;
        double v0 = p.alpha * s0, v1 = p.alpha * s1;
        if (p.vec2 && c + 1 < p.N) {
            if (p.beta != 0.0) {
                const double2 old = *reinterpret_cast<const double2*>(out);
                v0 = __fma_rn(p.beta, old.x, v0);
                v1 = __fma_rn(p.beta, old.y, v1);
            }
            *reinterpret_cast<double2*>(out) = make_double2(v0, v1);
        } else {
            out[0] = p.beta != 0.0 ? __fma_rn(p.beta, out[0], v0) : v0;
            if (c + 1 < p.N) out[1] = p.beta != 0.0 ? __fma_rn(p.beta, out[1], v1) : v1;
        }
    }
    cluster_sync_all();   // no block leaves while another reads its partial fragments
}

}  // namespace

// The cut of a shape: 0 = 32 x 16 tiles, else the cluster size (1, 2, 4 or 8)
// of the k-split kernel.  The costs are in MMAs of the busiest sub-partition,
// blocks spread evenly over the SMs: whole tiles cost their k-steps each;
// split blocks a quarter (an 8th, a 16th) of them, plus what their reductions
// and starts were measured to cost, about 0.3 per wave and 3 to 5 for the
// cluster's exchange.  Whole tiles win from about 10 waves on (64 x 8192 x 64:
// 70 us against 76; 2048^3: 15,681 against 15,706), splits below (700^3: 657
// against 699; 200 x 150 x 4000: 258 with clusters of four against 571).
// Eight blocks per cluster pay only while every block has an SM to itself
// (200 x 150 x 4000: 280, since clusters of eight do not spread evenly;
// 16 x 16 x 20000: 96 against 182).
int native_direct_cut(int64_t M, int64_t N, int64_t K, int sms) {
    const int64_t steps = (K + 3) / 4;
    const int64_t whole = ((M + 31) / 32) * ((N + 15) / 16), frags = ((M + 15) / 16) * ((N + 7) / 8);
    auto waves = [&](int64_t blocks) { return (double)((blocks + sms - 1) / sms); };
    double best = waves(whole) * (double)steps;
    int cut = 0;
    for (int size = 1; size <= 8; size *= 2) {
        if (size == 8 && frags * 8 > sms) break;
        const double w = waves(frags * size);
        const double c = w * (double)((steps + 4 * size - 1) / (4 * size)) + 0.3 * w +
                         (size == 1 ? 0.0 : 1.0 + 2.0 * (size == 2 ? 1 : 2));
        if (c < best) {
            best = c;
            cut = size;
        }
    }
    return cut;
}

// C = alpha op(A) op(B) + beta C for M, N, K > 0 and alpha != 0, every size
// below 2^31; any alignment and leading dimensions.  cut: as native_direct_cut
// gives it (-1: asked here); tile_limit > 0: only the first that many tiles or
// fragments of C (the tuner's timing proxy).
alp_status native_direct(int ta, int tb, int64_t M, int64_t N, int64_t K, double alpha,
                         const double* A, int64_t lda, const double* B, int64_t ldb, double beta,
                         double* C, int64_t ldc, cudaStream_t stream, int cut,
                         int64_t tile_limit) {
    DirectParams p;
    p.A = ta ? DirectOperand{A, 1, lda} : DirectOperand{A, lda, 1};
    p.B = tb ? DirectOperand{B, ldb, 1} : DirectOperand{B, 1, ldb};
    p.C = C;
    p.ldc = ldc;
    p.M = M;
    p.N = N;
    p.K = K;
    p.alpha = alpha;
    p.beta = beta;
    p.vec2 = (reinterpret_cast<uintptr_t>(C) & 15) == 0 && ldc % 2 == 0;
    if (cut < 0) cut = native_direct_cut(M, N, K, device_sm_count());
    p.tiles_m = cut ? (M + 15) / 16 : (M + 31) / 32;
    p.tiles_n = cut ? (N + 7) / 8 : (N + 15) / 16;
    int64_t tiles = p.tiles_m * p.tiles_n;
    if (tile_limit > 0) tiles = std::min(tiles, tile_limit);
    const int64_t blocks = tiles * std::max(cut, 1);
    if (blocks > 0x7fffffff) return ALP_ERR_UNSUPPORTED;
    if (cut <= 1) {
        auto kernel = cut ? dgemm_direct_split_kernel : dgemm_direct_kernel;
        kernel<<<(unsigned)blocks, 32 * kWarps, 0, stream>>>(p);
        return cuda_status(cudaGetLastError());
    }
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)blocks);
    lc.blockDim = dim3(32 * kWarps);
    lc.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cut;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    return cuda_status(cudaLaunchKernelEx(&lc, dgemm_direct_split_kernel, p));
}

}  // namespace alp

extern "C" int alp_native_cut(int64_t M, int64_t N, int64_t K, int sms) {
    if (M <= 0 || N <= 0 || K <= 0 || sms <= 0) return -1;
    return alp::native_direct_cut(M, N, K, sms);
}
