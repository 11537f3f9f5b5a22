// One launch that prepares both operands of an emulated GEMM: for every line
// (row of op(A), column of op(B)) the scale exponent and the digit or residue
// slices, K-major, from one read of the operand out of HBM.
//
// Lines that are contiguous in memory (rows of a row-major A, or of a B stored
// transposed) are walked by a warp each (K <= 2048) or a block each, the second
// pass served by L2.  Lines that are strided (columns of a row-major B) go
// through shared memory in strips of 32 bytes of columns (strips of 64 fill an
// SM with three blocks instead of four: 2048^2 42 us, not 35): a cluster of up
// to eight blocks holds a strip's whole k range (at most 1024 k per block), its
// blocks agree on the columns' maxima through distributed shared memory, and
// each splits its own part, so that no scan reads the operand beforehand.
//
// Bound by HBM for large operands (8 bytes read and 2 s written per element)
// and by launch latency for small ones: the scans, their initialisation and
// the splits were six launches of this chain.
#pragma once

#include "emul.cuh"
#include "emul_split.cuh"
#include "tc.cuh"

namespace alp {

constexpr int kPrepThreads = 256;
constexpr int kPrepWarps = kPrepThreads / 32;
constexpr int kPrepBlockK = 1024;                  // most k of a strip per block
constexpr int64_t kPrepMaxColK = 8 * kPrepBlockK;  // strided lines: clusters of at most eight
constexpr int64_t kPrepWarpRowK = 2048;            // contiguous lines up to this: one per warp

template <typename T>
struct PrepOperand {
    const T* X;           // null: not in this launch
    int64_t R, ldx;       // lines, and the leading dimension of their storage
    int32_t* exps;        // [R]
    __nv_bfloat16* out;   // [S][R][kpad]
    int cols;             // 1: line r is column r of X, else row r
    int blocks;           // of this operand in the launch
};

template <typename T>
struct PrepParams {
    PrepOperand<T> op[2];
    int64_t K, kpad;
    int block_k;          // k per block of a strip, a multiple of 128
    int known;            // 1: the exponents are given, 0: found and stored
    int* fill;            // words set to all ones (a schedule), may be null
    int64_t fill_words;
    int* err;
};

// Four consecutive elements of a line from k on, zeros past K.
template <typename T>
__device__ __forceinline__ void prep_load4(const T* __restrict__ x, int64_t k, int64_t K, bool vec,
                                           T (&a)[4]) {
    if (vec && k + 3 < K) {
        if constexpr (sizeof(T) == 8) {
            const double2 p = __ldg(reinterpret_cast<const double2*>(x + k));
            const double2 q = __ldg(reinterpret_cast<const double2*>(x + k + 2));
            a[0] = p.x;
            a[1] = p.y;
            a[2] = q.x;
            a[3] = q.y;
        } else {
            const float4 p = __ldg(reinterpret_cast<const float4*>(x + k));
            a[0] = p.x;
            a[1] = p.y;
            a[2] = p.z;
            a[3] = p.w;
        }
    } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) a[u] = k + u < K ? __ldg(x + k + u) : T(0);
    }
}

// (The sign is dropped in the high word: masked as 64 bits the compiler takes
// the magnitude with an FP64 operation, at a 64th of the integer rate.)
template <typename T>
__device__ __forceinline__ typename ScanKey<T>::type prep_key(T v) {
    if constexpr (sizeof(T) == 8)
        return ((uint64_t)(uint32_t)(__double2hiint(v) & 0x7FFFFFFF) << 32) |
               (uint32_t)__double2loint(v);
    else return ScanKey<T>::of((uint32_t)__float_as_int(v));
}

// The largest key of a contiguous line, TEAM threads (a warp or the block)
// with 4 strides of the line in flight each.
template <int TEAM, typename T>
__device__ __forceinline__ typename ScanKey<T>::type prep_line_max(
    const T* x, int64_t K, bool vec, int t, typename ScanKey<T>::type (*red)[kPrepWarps], int par) {
    using Key = typename ScanKey<T>::type;
    Key mx = 0;
#pragma unroll 1
    for (int64_t k0 = 4 * (int64_t)t; k0 < K; k0 += 16 * TEAM) {
        T a[4][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) prep_load4(x, k0 + (int64_t)q * 4 * TEAM, K, vec, a[q]);
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const Key y = prep_key(a[q][u]);
                mx = y > mx ? y : mx;
            }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const Key y = __shfl_xor_sync(0xffffffffu, mx, o);
        mx = y > mx ? y : mx;
    }
    if constexpr (TEAM > 32) {   // one slot set per line parity, one barrier per line
        if ((t & 31) == 0) red[par][t >> 5] = mx;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < TEAM / 32; ++w) mx = red[par][w] > mx ? red[par][w] : mx;
    }
    return mx;
}

template <int TEAM, int S, typename Sp, typename T>
__device__ __forceinline__ void prep_rows(const PrepParams<T>& p, const PrepOperand<T>& o,
                                          const Sp& sp, int block,
                                          typename ScanKey<T>::type (*red)[kPrepWarps]) {
    constexpr int kTeams = kPrepThreads / TEAM;
    const int t = threadIdx.x % TEAM;
    const int64_t plane = o.R * p.kpad;
    int par = 0;
    for (int64_t r = (int64_t)block * kTeams + threadIdx.x / TEAM; r < o.R;
         r += (int64_t)o.blocks * kTeams, par ^= 1) {
        const T* x = o.X + r * o.ldx;
        const bool vec = (reinterpret_cast<uintptr_t>(x) & 15) == 0;
        int e;
        if (p.known) {
            e = __ldg(o.exps + r);
        } else {
            const auto mx = prep_line_max<TEAM>(x, p.K, vec, t, red, par);
            e = frexp_exponent_of_bits(ScanKey<T>::to_double_bits(mx));
            if (t == 0) {
                o.exps[r] = e;
                if (mx >= ScanKey<T>::kInf) set_device_error(p.err, ALP_ERR_UNSUPPORTED);
            }
        }
        // the next stride's elements loaded before this one's are split
        T an[4];
        if (4 * (int64_t)t < p.kpad) prep_load4(x, 4 * (int64_t)t, p.K, vec, an);
#pragma unroll 1
        for (int64_t k = 4 * (int64_t)t; k < p.kpad; k += 4 * TEAM) {
            const T a[4] = {an[0], an[1], an[2], an[3]};
            if (k + 4 * TEAM < p.kpad) prep_load4(x, k + 4 * TEAM, p.K, vec, an);
            split4<S>(sp, a, e, o.out + r * p.kpad + k, plane);
        }
    }
}

// Strip geometry: a strip's columns, the row stride of its tile in shared
// memory (per column block_k + 12 elements) and the stride of the four k phases:
// element k = 4 q + i of a column sits at i * Q + q, so that the fill (16 rows of
// 2 column groups per warp) and the reads (consecutive q) are free of bank
// conflicts.
template <typename T>
constexpr int kPrepV = 16 / (int)sizeof(T);
constexpr int kPrepGroups = 2;   // 16-byte column groups per strip
template <typename T>
constexpr int kPrepStrip = kPrepGroups * kPrepV<T>;
template <typename T>
__host__ __device__ constexpr int prep_ld(int block_k) {
    return block_k + 12;
}
template <typename T>
__host__ __device__ constexpr int prep_q(int block_k) {
    return block_k / 4 + (sizeof(T) == 8 ? 2 : 4);
}
template <typename T>
constexpr size_t prep_smem(int block_k) {
    return sizeof(T) * kPrepStrip<T> * (size_t)prep_ld<T>(block_k);
}

// Fills the tile with rows kb0.. of the strip at column j0 (zeros past K and
// past the last column) and returns this thread's largest keys (columns
// j0 + V (lane & 3) + v).
template <typename T>
__device__ __forceinline__ void prep_fill(const PrepOperand<T>& o, int64_t K, int64_t j0,
                                          int64_t kb0, int rows, int block_k, T* tile,
                                          typename ScanKey<T>::type (&mx)[kPrepV<T>]) {
    constexpr int V = kPrepV<T>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cg = lane % kPrepGroups, rr = (32 / kPrepGroups) * warp + lane / kPrepGroups;
    const int ld = prep_ld<T>(block_k), Q = prep_q<T>(block_k);
    const int64_t j = j0 + V * cg;
    const T* x = o.X + kb0 * o.ldx + j;
    const bool vec = j + V <= o.R && (reinterpret_cast<uintptr_t>(x) & 15) == 0 &&
                     ((o.ldx * (int64_t)sizeof(T)) & 15) == 0;
    T* col = tile + V * cg * ld;
#pragma unroll
    for (int v = 0; v < V; ++v) mx[v] = 0;
    const int valid = (int)(K - kb0 < rows ? (K > kb0 ? K - kb0 : 0) : rows);
    constexpr int kStep = (32 / kPrepGroups) * kPrepWarps, kBatch = 8;   // rows per pass, passes in flight
#pragma unroll 1
    for (int r0 = rr; r0 < rows; r0 += kStep * kBatch) {
        T a[kBatch][V];
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const int r = r0 + b * kStep;
            const T* s = x + (int64_t)r * o.ldx;
            if (vec) {
                uint4 w = make_uint4(0u, 0u, 0u, 0u);
                if (r < valid) w = __ldg(reinterpret_cast<const uint4*>(s));
                if constexpr (sizeof(T) == 8) {
                    a[b][0] = __hiloint2double((int)w.y, (int)w.x);
                    a[b][1] = __hiloint2double((int)w.w, (int)w.z);
                } else {
                    a[b][0] = __uint_as_float(w.x);
                    a[b][1] = __uint_as_float(w.y);
                    a[b][2] = __uint_as_float(w.z);
                    a[b][3] = __uint_as_float(w.w);
                }
            } else {
#pragma unroll
                for (int v = 0; v < V; ++v)
                    a[b][v] = r < valid && j + v < o.R ? __ldg(s + v) : T(0);
            }
        }
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const int r = r0 + b * kStep;
            if (r < rows) {
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    col[v * ld + (r & 3) * Q + (r >> 2)] = a[b][v];
                    const auto y = prep_key(a[b][v]);
                    mx[v] = y > mx[v] ? y : mx[v];
                }
            }
        }
    }
}

// The columns' maxima over the whole cluster, in every thread t < strip width
// (column t), from the threads' keys: red [warps][strip], cmax [strip].  All
// threads call it; it ends the fill (a block barrier), and the caller passes a
// cluster barrier (size > 1) before its block exits.
template <typename T>
__device__ __forceinline__ typename ScanKey<T>::type prep_column_max(
    typename ScanKey<T>::type (&mx)[kPrepV<T>], typename ScanKey<T>::type* red,
    typename ScanKey<T>::type* cmax, uint32_t size) {
    using Key = typename ScanKey<T>::type;
    constexpr int V = kPrepV<T>, W = kPrepStrip<T>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int v = 0; v < V; ++v) {
#pragma unroll
        for (int o = kPrepGroups; o <= 16; o <<= 1) {
            const Key y = __shfl_xor_sync(0xffffffffu, mx[v], o);
            mx[v] = y > mx[v] ? y : mx[v];
        }
        if (lane < kPrepGroups) red[warp * W + V * lane + v] = mx[v];
    }
    __syncthreads();
    Key m = 0;
    const int t = threadIdx.x;
    if (t < W) {
#pragma unroll
        for (int w = 0; w < kPrepWarps; ++w) m = red[w * W + t] > m ? red[w * W + t] : m;
        cmax[t] = m;
    }
    if (size > 1) {
        cluster_sync_all();
        if (t < W)
            for (uint32_t q = 0; q < size; ++q) {
                const uint32_t a = cluster_addr(&cmax[t], q);
                Key y;
                if constexpr (sizeof(Key) == 8)
                    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(y) : "r"(a) : "memory");
                else
                    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(y) : "r"(a) : "memory");
                m = y > m ? y : m;
            }
    }
    return m;
}

template <int S, typename Sp, typename T>
__device__ __forceinline__ void prep_cols(const PrepParams<T>& p, const PrepOperand<T>& o,
                                          const Sp& sp, int block, T* tile,
                                          typename ScanKey<T>::type* red,
                                          typename ScanKey<T>::type* cmax, int* sexp) {
    constexpr int W = kPrepStrip<T>;
    const uint32_t rank = cluster_ctarank(), size = cluster_nctarank();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t j0 = (int64_t)(block / (int)size) * W, kb0 = (int64_t)rank * p.block_k;
    const int rows = (int)min((int64_t)p.block_k, max(p.kpad - kb0, (int64_t)0));
    typename ScanKey<T>::type mx[kPrepV<T>];
    prep_fill(o, p.K, j0, kb0, rows, p.block_k, tile, mx);
    if (p.known) {
        if (threadIdx.x < W)
            sexp[threadIdx.x] = j0 + threadIdx.x < o.R ? __ldg(o.exps + j0 + threadIdx.x) : 0;
    } else {
        const auto m = prep_column_max<T>(mx, red, cmax, size);
        if (threadIdx.x < W) {
            const int e = frexp_exponent_of_bits(ScanKey<T>::to_double_bits(m));
            sexp[threadIdx.x] = e;
            if (rank == 0 && j0 + threadIdx.x < o.R) {
                o.exps[j0 + threadIdx.x] = e;
                if (m >= ScanKey<T>::kInf) set_device_error(p.err, ALP_ERR_UNSUPPORTED);
            }
        }
    }
    __syncthreads();
    const int ld = prep_ld<T>(p.block_k), Q = prep_q<T>(p.block_k);
    const int64_t plane = o.R * p.kpad;
    // warp w takes column w % W and every (warps / W)-th 128 k of it
    for (int c = warp % W; c < W; c += kPrepWarps) {
        const int64_t j = j0 + c;
        if (j >= o.R) break;
        const int e = sexp[c];
        const T* col = tile + c * ld;
#pragma unroll 1
        for (int k = 4 * lane + 128 * (warp / W); k < rows;
             k += 128 * (kPrepWarps > W ? kPrepWarps / W : 1)) {
            const int q = k >> 2;
            const T a[4] = {col[q], col[Q + q], col[2 * Q + q], col[3 * Q + q]};
            split4<S>(sp, a, e, o.out + j * p.kpad + kb0 + k, plane);
        }
    }
    if (size > 1 && !p.known) cluster_sync_all();   // cmax read by the whole cluster
}

template <typename T, int S, typename Sp>
__global__ void __launch_bounds__(kPrepThreads, 4)
    emul_prep_kernel(const __grid_constant__ PrepParams<T> p, const Sp sp) {
    using Key = typename ScanKey<T>::type;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ Key red[kPrepWarps * (kPrepStrip<T> > 2 ? kPrepStrip<T> : 2)];
    __shared__ Key cmax[kPrepStrip<T>];
    __shared__ int sexp[kPrepStrip<T>];
    pdl_launch();
    for (int64_t i = (int64_t)blockIdx.x * kPrepThreads + threadIdx.x; i < p.fill_words;
         i += (int64_t)gridDim.x * kPrepThreads)
        p.fill[i] = -1;
    const bool second = (int)blockIdx.x >= p.op[0].blocks;
    const PrepOperand<T>& o = p.op[second ? 1 : 0];
    const int block = (int)blockIdx.x - (second ? p.op[0].blocks : 0);
    if (o.cols)
        prep_cols<S>(p, o, sp, block, reinterpret_cast<T*>(smem_raw), red, cmax, sexp);
    else if (p.K <= kPrepWarpRowK)
        prep_rows<32, S>(p, o, sp, block, reinterpret_cast<Key(*)[kPrepWarps]>(red));
    else
        prep_rows<kPrepThreads, S>(p, o, sp, block, reinterpret_cast<Key(*)[kPrepWarps]>(red));
}

// The cut of a launch: cluster size and k per block of the strips (the whole k
// range while it fits a block: it is loaded in one go either way, and a second
// block only adds the cluster's barriers; but at least a block on every second
// SM, of 128 k or more), blocks per operand (multiples of the cluster size).
// Against two blocks per SM as the aim: CRT 1024^3 68.0 -> 64.0 us, 768^3 41.4
// -> 39.5, with the automatic count 95.5 -> 90.4 and 67.4 -> 63.8, FP32 45.5 -> 43.6.
template <typename T>
inline int prep_cut(PrepParams<T>& p, int sms) {
    int64_t strips = 0;
    for (const auto& o : p.op)
        if (o.X && o.cols) strips += (o.R + kPrepStrip<T> - 1) / kPrepStrip<T>;
    int size = 1;
    p.block_k = 128;
    if (strips) {
        auto per = [&](int c) { return (int)(((p.kpad + c - 1) / c + 127) / 128 * 128); };
        while (size < 8 && (per(size) > kPrepBlockK ||
                            (2 * strips * size < (int64_t)sms && per(size) > 128)))
            size *= 2;
        p.block_k = per(size);
    }
    for (auto& o : p.op) {
        int64_t b;
        if (!o.X) {
            b = 0;   // not in this launch
        } else if (o.cols) {
            b = (o.R + kPrepStrip<T> - 1) / kPrepStrip<T> * size;
        } else {
            b = p.K <= kPrepWarpRowK ? (o.R + kPrepWarps - 1) / kPrepWarps : o.R;
            b = b < (int64_t)sms * 12 ? b : (int64_t)sms * 12;   // four waves of 3 per SM
            b = (b + size - 1) / size * size;
        }
        o.blocks = (int)b;
    }
    return size;
}

// Whether strided lines go through the strips: their k must fit a cluster, and
// the operand must be small enough that launches count.  A strip's load, its
// maxima and its split follow one another in each block, so that at 4096^2 a
// scan and a split kernel of their own, each at the HBM rate, take 128 us
// against 145 (2048^2: 41 and three launches against 35; float, with 6 bytes
// written per element instead of 30, the strips win up to 5000^2).  Short lines
// leave a block little to overlap that chain with, so that many of them are too
// large as well (whole calls with M = 64, strips and separate, us; N x K is the
// strided operand): 8 digits 24576 x 64 166 and 168, 32768 x 64 204 and 201, 131072
// x 64 748 and 678; 32768 x 192 241 and 242, 61000 x 136 434 and 424; float, 3 digits
// 49152 x 64 94 and 96, 65536 x 64 107.5 and 106.5, 131072 x 64 206 and 187, but 131072
// x 256 255 and 268.  With the automatic count's statistics in the strips as well
// (stats), clusters of eight blocks cost more than launches from a smaller size on:
// 1024 x 1024 x 8192, A and B strided, 456 and 412, 800 x 800 x 8190 394 and 378, 700 x
// 700 x 8190 301 and 306.
template <typename T>
inline bool prep_in_strips(int64_t R, int64_t K, bool stats = false) {
    if (stats && K > 4 * kPrepBlockK && R * K > int64_t(6) << 20) return false;
    const int64_t strips = (R + kPrepStrip<T> - 1) / kPrepStrip<T>;
    return K <= kPrepMaxColK &&
           R * K <= (sizeof(T) == 8 ? int64_t(1) << 23 : int64_t(1) << 25) &&
           strips <= (K <= 128 ? 6144 : sizeof(T) == 8 ? 8192 : int64_t(1) << 22);
}

// Launches `kernel` (of these roles) with the cut of p's operands.
template <typename T, typename Kernel, typename Arg>
alp_status launch_prep_kernel(Kernel kernel, PrepParams<T> p, cudaStream_t st, const Arg& arg) {
    const int size = prep_cut(p, device_sm_count());
    const bool cols = p.op[0].cols || p.op[1].cols;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)prep_smem<T>(kPrepBlockK));
    if (e != cudaSuccess) return cuda_status(e);
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)(p.op[0].blocks + p.op[1].blocks));
    lc.blockDim = dim3(kPrepThreads);
    lc.dynamicSmemBytes = cols ? prep_smem<T>(p.block_k) : 0;
    lc.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)size;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    return cuda_status(cudaLaunchKernelEx(&lc, kernel, p, arg));
}

template <typename T, int S, typename Sp>
alp_status launch_prep(const PrepParams<T>& p, const Sp& sp, cudaStream_t st) {
    return launch_prep_kernel(emul_prep_kernel<T, S, Sp>, p, st, sp);
}

}  // namespace alp
