// Batched variable-size native FP64 GEMM: thousands of independent problems
// C_p = alpha_p A_p B_p + beta_p C_p in one persistent launch.
//
// 1. A one-block plan kernel orders the problems by K bucket, longest first,
//    and by tile class within it (row and column tile of 32, 64 or 128, from M
//    and N), and writes the prefix sum of their unit counts: the device work
//    list.  Everything it reads is device memory, so the call is
//    stream-ordered and capturable in a CUDA graph.
// 2. In a persistent kernel every warp on its own takes units from an atomic
//    counter, a unit being one 16 x 16 block of one problem's C over the whole
//    of its k, finds the problem by binary search in the prefix array, and
//    runs it with register-direct DMMA fragments (native_direct.cuh).
//
// The launch is bound by the FP64 MMA rate, so what counts is that no MMA is
// spent on padding and that all sub-partitions end together: 16 x 8 fragments
// outside a problem are skipped, and units are small and end with the
// shortest k.  4096 problems of 16..1024 (1.11e11 flops: 101.3 ms at the MMA
// rate, 106.9 with whole fragments): 108.6 ms; the class table's default tiles,
// one 8-warp block per SM, took 153.6.
//
// The class -> (bm, bn, bk) table is runtime state (alp_batched_set_class_config).
#include <algorithm>
#include <cstdlib>
#include <mutex>

#include "alp_ext.h"
#include "native_direct.cuh"

namespace alp {

namespace {

constexpr int kClasses = 9;           // 3 row-tile x 3 column-tile sizes
constexpr int kKBuckets = 16;         // floor(log2 K) buckets, longest first
constexpr int kBatchedThreads = 128;  // warps work alone; four per block, one per sub-partition
constexpr int kUnit = 16;             // rows and columns of C per unit of work
constexpr int kPlanThreads = 1024;

struct ClassTable {
    int bm[kClasses], bn[kClasses], bk[kClasses];
};

std::mutex g_bmu;
ClassTable g_table = {
    {32, 32, 32, 64, 64, 64, 128, 128, 128},
    {32, 64, 128, 32, 64, 128, 32, 64, 128},
    {32, 32, 16, 32, 16, 16, 16, 16, 16}};

ClassTable current_table() {
    std::lock_guard<std::mutex> lk(g_bmu);
    return g_table;
}

__host__ __device__ __forceinline__ int size_bucket(int64_t v) { return v <= 32 ? 0 : v <= 64 ? 1 : 2; }
__host__ __device__ __forceinline__ int class_of(int64_t M, int64_t N) {
    return size_bucket(M) * 3 + size_bucket(N);
}

struct BatchArgs {
    int64_t count;
    const int64_t *M, *N, *K, *lda, *ldb, *ldc;
    const double *alpha, *beta;
    const double* const* A;
    const double* const* B;
    double* const* C;
};

struct Plan {              // device workspace
    int32_t* key;          // [count] sort key per problem (-1: nothing to do)
    int32_t* order;        // [count] problem ids in (K bucket desc, class) order
    int64_t* prefix;       // [count + 1] exclusive unit prefix over `order`
    int64_t* meta;         // [0] valid problems, [1] total units
    unsigned long long* counter;   // unit counter of the persistent kernel
};

__host__ __device__ __forceinline__ int64_t units_of(int64_t M, int64_t N) {
    return ((M + kUnit - 1) / kUnit) * ((N + kUnit - 1) / kUnit);
}

__global__ void __launch_bounds__(kPlanThreads) batched_plan_kernel(BatchArgs a, Plan pl) {
    __shared__ int cnt[kClasses * kKBuckets];
    __shared__ int base[kClasses * kKBuckets];
    __shared__ int64_t chunk_sum[kPlanThreads];
    __shared__ int64_t carry;
    const int tid = threadIdx.x;
    for (int i = tid; i < kClasses * kKBuckets; i += kPlanThreads) cnt[i] = 0;
    __syncthreads();
    for (int64_t p = tid; p < a.count; p += kPlanThreads) {
        const int64_t M = a.M[p], N = a.N[p];
        int64_t K = a.K[p];
        if (a.alpha[p] == 0.0) K = 0;
        int key = -1;
        if (M > 0 && N > 0) {
            const int kb = K > 0 ? 63 - __clzll((long long)K) : 0;
            key = (kKBuckets - 1 - (kb < kKBuckets ? kb : kKBuckets - 1)) * kClasses + class_of(M, N);
            atomicAdd(&cnt[key], 1);
        }
        pl.key[p] = key;
    }
    __syncthreads();
    if (tid == 0) {
        int run = 0;
        for (int i = 0; i < kClasses * kKBuckets; ++i) {
            base[i] = run;
            run += cnt[i];
        }
        pl.meta[0] = run;
    }
    __syncthreads();
    for (int64_t p = tid; p < a.count; p += kPlanThreads) {
        const int key = pl.key[p];
        if (key >= 0) pl.order[atomicAdd(&base[key], 1)] = (int32_t)p;
    }
    __syncthreads();
    // exclusive prefix of unit counts along `order`, 1024 entries at a time
    const int64_t nvalid = pl.meta[0];
    if (tid == 0) carry = 0;
    __syncthreads();
    for (int64_t c0 = 0; c0 < nvalid; c0 += kPlanThreads) {
        const int64_t pos = c0 + tid;
        int64_t units = 0;
        if (pos < nvalid) {
            const int32_t p = pl.order[pos];
            units = units_of(a.M[p], a.N[p]);
        }
        chunk_sum[tid] = units;
        __syncthreads();
        for (int off = 1; off < kPlanThreads; off <<= 1) {   // inclusive Hillis-Steele scan
            const int64_t v = tid >= off ? chunk_sum[tid - off] : 0;
            __syncthreads();
            chunk_sum[tid] += v;
            __syncthreads();
        }
        if (pos < nvalid) pl.prefix[pos] = carry + chunk_sum[tid] - units;
        __syncthreads();
        if (tid == kPlanThreads - 1) carry += chunk_sum[tid];
        __syncthreads();
    }
    if (tid == 0) {
        pl.prefix[nvalid] = carry;
        pl.meta[1] = carry;
        *pl.counter = 0ull;
    }
}

__global__ void __launch_bounds__(kBatchedThreads, 5)
    batched_persistent_kernel(const __grid_constant__ BatchArgs a, const __grid_constant__ Plan pl,
                              const __grid_constant__ ClassTable tab) {
    const int lane = threadIdx.x & 31;
    const int64_t total = pl.meta[1];
    const int64_t nvalid = pl.meta[0];
    while (true) {
        int64_t t = 0;
        if (lane == 0) t = (int64_t)atomicAdd(pl.counter, 1ull);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= total) break;
        // position: last pos with prefix[pos] <= t
        int64_t lo = 0, hi = nvalid - 1;
        while (lo < hi) {
            const int64_t mid = (lo + hi + 1) >> 1;
            if (pl.prefix[mid] <= t) lo = mid;
            else hi = mid - 1;
        }
        const int32_t p = pl.order[lo];
        const int64_t M = a.M[p], N = a.N[p];
        const double alpha = a.alpha[p];
        const int64_t K = alpha == 0.0 ? 0 : a.K[p];
        // units run down the rows of a tile-row (bm of the problem's class)
        // before moving one unit-column right, for reuse of B's columns
        const int64_t un = (N + kUnit - 1) / kUnit, um = (M + kUnit - 1) / kUnit;
        const int64_t strip = tab.bm[class_of(M, N)] / kUnit;
        const int64_t local = t - pl.prefix[lo];
        const int64_t first = local / (strip * un) * strip;
        const int64_t rows = min(um - first, strip);
        const int64_t rem = local % (strip * un);
        const int64_t r0 = (first + rem % rows) * kUnit, c0 = rem / rows * kUnit;
        double* C = a.C[p];
        const int64_t ldc = a.ldc[p];
        Acc<2, 4> acc;
        acc.zero();
        mma_direct<1, 2>(DirectOperand{a.A[p], a.lda[p], 1}, DirectOperand{a.B[p], 1, a.ldb[p]}, M,
                         N, K, r0, c0, 0, (K + 3) >> 2, lane, acc);
        const bool vec2 = (reinterpret_cast<uintptr_t>(C) & 15) == 0 && ldc % 2 == 0;
        epilogue<2, 4>(acc, C, ldc, M, N, r0, c0, alpha, a.beta[p], vec2, lane);
    }
}

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

struct PlanLayout {
    size_t off_key, off_order, off_prefix, off_meta, off_counter, bytes;
};

PlanLayout plan_layout(int64_t count) {
    PlanLayout L;
    size_t off = 0;
    L.off_key = off; off += up256((size_t)count * 4);
    L.off_order = off; off += up256((size_t)count * 4);
    L.off_prefix = off; off += up256((size_t)(count + 1) * 8);
    L.off_meta = off; off += 256;
    L.off_counter = off; off += 256;
    L.bytes = off;
    return L;
}

// The persistent kernel for `units` units on `sms` SMs, as many blocks as fit.
alp_status launch_persistent(const BatchArgs& a, const Plan& pl, const ClassTable& tab,
                             int64_t units, int sms, cudaStream_t stream) {
    int occ = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, batched_persistent_kernel,
                                                  kBatchedThreads, 0);
    if (occ < 1) occ = 1;
    const int64_t grid = std::min<int64_t>((int64_t)sms * occ, (units + 3) / 4);
    batched_persistent_kernel<<<(unsigned)grid, kBatchedThreads, 0, stream>>>(a, pl, tab);
    return cuda_status(cudaGetLastError());
}

}  // namespace

// Launches plan + persistent kernel for the whole batch on `sms` SMs, with the
// work list in `workspace` (256-byte aligned, plan_layout(count).bytes).
alp_status batched_launch(const BatchArgs& a, const int64_t* hM, const int64_t* hN,
                          void* workspace, cudaStream_t stream, int sms) {
    const ClassTable tab = current_table();
    const PlanLayout L = plan_layout(a.count);
    char* ws = static_cast<char*>(workspace);
    Plan pl;
    pl.key = reinterpret_cast<int32_t*>(ws + L.off_key);
    pl.order = reinterpret_cast<int32_t*>(ws + L.off_order);
    pl.prefix = reinterpret_cast<int64_t*>(ws + L.off_prefix);
    pl.meta = reinterpret_cast<int64_t*>(ws + L.off_meta);
    pl.counter = reinterpret_cast<unsigned long long*>(ws + L.off_counter);
    // grid size from the host copies (performance only: the persistent loop
    // covers any number of units)
    int64_t units = 0;
    for (int64_t p = 0; p < a.count; ++p)
        if (hM[p] > 0 && hN[p] > 0) units += units_of(hM[p], hN[p]);
    batched_plan_kernel<<<1, kPlanThreads, 0, stream>>>(a, pl);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_status(e);
    if (units == 0) return ALP_OK;
    return launch_persistent(a, pl, tab, units, sms, stream);
}

}  // namespace alp

using namespace alp;

namespace {
bool class_config_ok(int bm, int bn, int bk) {
    auto ok = [](int v) { return v == 32 || v == 64 || v == 128; };
    return ok(bm) && ok(bn) && (bk == 16 || bk == 32 || bk == 64) &&
           2 * (bm + bn) * bk * 8 <= kSmemLimit;
}

alp_status fill_args(BatchArgs& a, int64_t count, const int64_t* dM, const int64_t* dN,
                     const int64_t* dK, const double* dalpha, const double* const* dA,
                     const int64_t* dlda, const double* const* dB, const int64_t* dldb,
                     const double* dbeta, double* const* dC, const int64_t* dldc) {
    if (!dM || !dN || !dK || !dalpha || !dA || !dlda || !dB || !dldb || !dbeta || !dC || !dldc)
        return ALP_ERR_INVALID_ARG;
    a.count = count;
    a.M = dM; a.N = dN; a.K = dK; a.alpha = dalpha; a.beta = dbeta;
    a.A = dA; a.B = dB; a.C = dC; a.lda = dlda; a.ldb = dldb; a.ldc = dldc;
    return ALP_OK;
}

alp_status check_host_sizes(int64_t count, const int64_t* hM, const int64_t* hN,
                            const int64_t* hK) {
    if (count < 0 || count > 0x7fffffff) return ALP_ERR_INVALID_ARG;
    if (count > 0 && (!hM || !hN || !hK)) return ALP_ERR_INVALID_ARG;
    for (int64_t p = 0; p < count; ++p)
        if (hM[p] < 0 || hN[p] < 0 || hK[p] < 0) return ALP_ERR_INVALID_ARG;
    return ALP_OK;
}

struct BatchedGraph {
    cudaGraph_t graph;
    cudaGraphExec_t exec;
};
}  // namespace

extern "C" {

size_t alp_gemm_batched_workspace(int64_t count, const int64_t* hM, const int64_t* hN,
                                  const int64_t* hK) {
    if (check_host_sizes(count, hM, hN, hK) != ALP_OK) return 0;
    return plan_layout(count).bytes;
}

alp_status alp_gemm_batched_varsize(int64_t count, const int64_t* dM, const int64_t* dN,
                                    const int64_t* dK, const double* dalpha,
                                    const double* const* dA, const int64_t* dlda,
                                    const double* const* dB, const int64_t* dldb,
                                    const double* dbeta, double* const* dC,
                                    const int64_t* dldc, const int64_t* hM,
                                    const int64_t* hN, const int64_t* hK, void* workspace,
                                    size_t workspace_bytes, void* stream) {
    alp_status st = check_host_sizes(count, hM, hN, hK);
    if (st != ALP_OK) return st;
    if (count == 0) return ALP_OK;
    BatchArgs a;
    if ((st = fill_args(a, count, dM, dN, dK, dalpha, dA, dlda, dB, dldb, dbeta, dC, dldc)) !=
        ALP_OK)
        return st;
    if (!workspace || workspace_bytes < plan_layout(count).bytes || ((uintptr_t)workspace & 255))
        return ALP_ERR_WORKSPACE;
    return batched_launch(a, hM, hN, workspace, reinterpret_cast<cudaStream_t>(stream),
                          device_sm_count());
}

alp_status alp_batched_set_class_config(int cls, int bm, int bn, int bk) {
    if (cls < 0 || cls >= kClasses || !class_config_ok(bm, bn, bk)) return ALP_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lk(g_bmu);
    g_table.bm[cls] = bm;
    g_table.bn[cls] = bn;
    g_table.bk[cls] = bk;
    return ALP_OK;
}

alp_status alp_batched_get_class_config(int cls, int* bm, int* bn, int* bk) {
    if (cls < 0 || cls >= kClasses || !bm || !bn || !bk) return ALP_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lk(g_bmu);
    *bm = g_table.bm[cls];
    *bn = g_table.bn[cls];
    *bk = g_table.bk[cls];
    return ALP_OK;
}

int alp_batched_class_of(int64_t M, int64_t N) { return class_of(M, N); }

alp_status alp_batched_graph_create(int64_t count, const int64_t* dM, const int64_t* dN,
                                    const int64_t* dK, const double* dalpha,
                                    const double* const* dA, const int64_t* dlda,
                                    const double* const* dB, const int64_t* dldb,
                                    const double* dbeta, double* const* dC,
                                    const int64_t* dldc, const int64_t* hM,
                                    const int64_t* hN, const int64_t* hK, void* workspace,
                                    size_t workspace_bytes, void** graph_out) {
    if (!graph_out) return ALP_ERR_INVALID_ARG;
    *graph_out = nullptr;
    // one-time per-device set-up (error word, SM count) must not happen
    // inside the capture
    if (!device_error_word() || device_sm_count() < 1) return ALP_ERR_CUDA;
    cudaStream_t cs;
    if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) return ALP_ERR_CUDA;
    BatchedGraph* g = new BatchedGraph{nullptr, nullptr};
    alp_status st = ALP_OK;
    if (cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
        st = ALP_ERR_CUDA;
    } else {
        st = alp_gemm_batched_varsize(count, dM, dN, dK, dalpha, dA, dlda, dB, dldb, dbeta, dC,
                                      dldc, hM, hN, hK, workspace, workspace_bytes, cs);
        cudaGraph_t graph = nullptr;
        const cudaError_t e = cudaStreamEndCapture(cs, &graph);
        if (st == ALP_OK && e != cudaSuccess) st = ALP_ERR_CUDA;
        g->graph = graph;
        if (st == ALP_OK && cudaGraphInstantiate(&g->exec, graph, 0) != cudaSuccess)
            st = ALP_ERR_CUDA;
    }
    cudaStreamDestroy(cs);
    if (st != ALP_OK) {
        if (g->exec) cudaGraphExecDestroy(g->exec);
        if (g->graph) cudaGraphDestroy(g->graph);
        delete g;
        return st;
    }
    *graph_out = g;
    return ALP_OK;
}

alp_status alp_batched_graph_launch(void* graph, void* stream) {
    if (!graph) return ALP_ERR_INVALID_ARG;
    BatchedGraph* g = static_cast<BatchedGraph*>(graph);
    return cuda_status(cudaGraphLaunch(g->exec, reinterpret_cast<cudaStream_t>(stream)));
}

alp_status alp_batched_graph_destroy(void* graph) {
    if (!graph) return ALP_OK;
    BatchedGraph* g = static_cast<BatchedGraph*>(graph);
    cudaGraphExecDestroy(g->exec);
    cudaGraphDestroy(g->graph);
    delete g;
    return ALP_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Batched GEMM without a caller-provided workspace.
//
// Some callers cannot allocate device memory at the point where they issue
// the GEMM: frameworks whose device memory is owned by their own pool
// allocator, and real-time or long-running loops that must not take the
// allocator's locks or risk the implicit device synchronisation of
// cudaMalloc / cudaFree.  For them this entry point keeps the work list of
// the persistent kernel in one file-scope device array instead of a
// workspace.  The array is part of the library image: every GPU that loads
// the library holds these kNoAllocScratchBytes until the process exits.
// ---------------------------------------------------------------------------
namespace {
constexpr size_t kNoAllocScratchBytes = size_t(1) << 20;   // 1 MiB: up to 65,000 problems
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

std::mutex g_noalloc_mu;
void* g_noalloc_ptr[64];   // device address of g_noalloc_scratch per device (nullptr: not set up)
int g_noalloc_sms[64];     // SM count per device

// Device address of the scratch array on the current device and its SM count.
// The first call on a device looks both up (cudaGetSymbolAddress and an
// attribute query, neither of which allocates); later calls reuse them.
alp_status noalloc_scratch(void** out, int* sms) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return ALP_ERR_CUDA;
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return ALP_ERR_CUDA;
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            n < 1)
            return ALP_ERR_CUDA;
        g_noalloc_sms[dev] = n;
        g_noalloc_ptr[dev] = p;
    }
    *out = g_noalloc_ptr[dev];
    *sms = g_noalloc_sms[dev];
    return ALP_OK;
}
}  // namespace

extern "C" alp_status alp_gemm_batched_varsize_noalloc(
    int64_t count, const int64_t* dM, const int64_t* dN, const int64_t* dK, const double* dalpha,
    const double* const* dA, const int64_t* dlda, const double* const* dB, const int64_t* dldb,
    const double* dbeta, double* const* dC, const int64_t* dldc, const int64_t* hM,
    const int64_t* hN, const int64_t* hK, void* stream) {
    alp_status st = check_host_sizes(count, hM, hN, hK);
    if (st != ALP_OK) return st;
    if (count == 0) return ALP_OK;
    if (plan_layout(count).bytes > kNoAllocScratchBytes) return ALP_ERR_WORKSPACE;   // too many problems
    BatchArgs a;
    if ((st = fill_args(a, count, dM, dN, dK, dalpha, dA, dlda, dB, dldb, dbeta, dC, dldc)) !=
        ALP_OK)
        return st;
    void* scratch = nullptr;
    int sms = 0;
    if ((st = noalloc_scratch(&scratch, &sms)) != ALP_OK) return st;
    // The same launch as alp_gemm_batched_varsize with the scratch array as its
    // workspace (256-byte aligned, as a workspace must be).  The plan kernel
    // rewrites every part of it that it later reads (keys, order, prefix sums,
    // counts, and the unit counter it sets to 0), so the previous call's
    // contents need no clearing.
    return batched_launch(a, hM, hN, scratch, reinterpret_cast<cudaStream_t>(stream), sms);
}
