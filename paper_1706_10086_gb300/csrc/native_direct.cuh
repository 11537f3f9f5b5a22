// Warp-level building block of the FP64 GEMM kernels that read their operands
// straight into registers (native_direct.cu, batched.cu).
//
// On this GPU one m16n8k4 FP64 MMA holds its SM sub-partition for about 1170
// clocks (0.4375 FMA per clock and sub-partition: 1.098 TFLOP/s over 608 of
// them, measured), longer than a load from L2 takes to arrive.  What bounds an
// FP64 GEMM here is therefore only how evenly its MMAs are spread over the
// sub-partitions and how few of them are spent on padding; operand traffic is
// small (a 32 x 32 tile moves 2 KB per 2340 clocks).  So the operands skip
// shared memory: each lane loads its own fragment elements, kDirectDepth
// k-steps ahead, with no alignment, stride or transposition rule, and
// fragments that lie outside M x N are not multiplied.
#pragma once

#include "native.cuh"

namespace alp {

// op(X) by its strides in elements: element (row, k) of op(A) at
// p[row * outer + k * inner], element (k, col) of op(B) at
// p[col * outer + k * inner].
struct DirectOperand {
    const double* p;
    int64_t outer, inner;
};

constexpr int kDirectDepth = 4;   // k-steps (of 4) in flight per warp

// acc += op(A)[r0.., 4 s0 .. ) op(B): k-steps s0..s1-1 (each of 4 k; k >= K
// contributes zeros) of the FM x FN fragments (16 x 8 each) at row r0, column
// c0.  Rows past M and columns past N are read from the last valid row or
// column and only feed results that are not stored; fragments wholly outside
// are skipped.  The order of the MMAs over k is ascending, as in mma_stage, so
// a sum over all k-steps has the same bits as the shared-memory kernels'.
template <int FM, int FN>
__device__ __forceinline__ void mma_direct(const DirectOperand& A, const DirectOperand& B,
                                           int64_t M, int64_t N, int64_t K, int64_t r0, int64_t c0,
                                           int64_t s0, int64_t s1, int lane,
                                           Acc<2 * FM, 2 * FN>& acc) {
    const int g = lane >> 2, t = lane & 3;
    const int fm = r0 >= M ? 0 : (int)min((int64_t)FM, (M - r0 + 15) >> 4);
    const int fn = c0 >= N ? 0 : (int)min((int64_t)FN, (N - c0 + 7) >> 3);
    if (fm == 0 || fn == 0 || s0 >= s1) return;
    const double* pa[FM][2];
    const double* pb[FN];
#pragma unroll
    for (int i = 0; i < FM; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int64_t r = min(r0 + 16 * i + 8 * h + g, M - 1);
            pa[i][h] = A.p + r * A.outer + (4 * s0 + t) * A.inner;
        }
#pragma unroll
    for (int j = 0; j < FN; ++j) {
        const int64_t c = min(c0 + 8 * j + g, N - 1);
        pb[j] = B.p + c * B.outer + (4 * s0 + t) * B.inner;
    }
    const int64_t da = 4 * A.inner, db = 4 * B.inner;
    // this lane's k-steps with k = 4 s + t < K (the last may be one fewer)
    const int64_t klim = (K - t + 3) >> 2;
    const int n = (int)(s1 - s0);
    const int nl = (int)(min(s1, klim) - s0);
    double a[kDirectDepth][FM][2], b[kDirectDepth][FN];
    auto load = [&](int s, double (&x)[FM][2], double (&y)[FN]) {
        const bool ok = s < nl;
#pragma unroll
        for (int i = 0; i < FM; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                x[i][h] = ok ? __ldg(pa[i][h]) : 0.0;
                pa[i][h] += da;
            }
#pragma unroll
        for (int j = 0; j < FN; ++j) {
            y[j] = ok ? __ldg(pb[j]) : 0.0;
            pb[j] += db;
        }
    };
#pragma unroll
    for (int d = 0; d < kDirectDepth; ++d) load(d, a[d], b[d]);
    for (int s = 0; s < n; s += kDirectDepth) {
#pragma unroll
        for (int d = 0; d < kDirectDepth; ++d) {
            if (s + d >= n) break;
#pragma unroll
            for (int i = 0; i < FM; ++i)
#pragma unroll
                for (int j = 0; j < FN; ++j)
                    if (i < fm && j < fn)
                        dmma_16x8x4(acc.c[i][j], a[d][i][0], a[d][i][1], b[d][j]);
            load(s + d + kDirectDepth, a[d], b[d]);
        }
    }
}

}  // namespace alp
