// C-ABI entry points, argument validation, per-device state (error word, SM
// count, tensor-map encoder) and config selection for alp_gemm_f64.
#include <cudaTypedefs.h>

#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>

#include "alp_internal.cuh"
#include "alp_ext.h"
#include "native_cfg.h"
#include "emul.cuh"

namespace alp {

alp_status native_launch(const alp_config& cfg, bool use_tma, int64_t M, int64_t N, int64_t K,
                         double alpha, const double* A, int64_t lda, const double* B,
                         int64_t ldb, double beta, double* C, int64_t ldc, cudaStream_t stream,
                         int inject_skip_kt, int64_t grid_limit);
alp_status native_transpose(const double* X, int64_t R, int64_t Cn, int64_t ldx, double* out,
                            int64_t ldo, cudaStream_t stream);
alp_status native_scale(int64_t M, int64_t N, double beta, double* C, int64_t ldc,
                        cudaStream_t stream);
alp_status native_direct(int ta, int tb, int64_t M, int64_t N, int64_t K, double alpha,
                         const double* A, int64_t lda, const double* B, int64_t ldb, double beta,
                         double* C, int64_t ldc, cudaStream_t stream, int cut = -1,
                         int64_t tile_limit = 0);
// tune.cu: the config a call without one runs with; false when there is none.
bool tuned_config(int64_t M, int64_t N, int64_t K, alp_path path, alp_config* out,
                  cudaStream_t stream);

// ----------------------------------------------------------------------------
// Per-device state.
// ----------------------------------------------------------------------------
namespace {
constexpr int kMaxDevices = 64;
// g_mu guards the set-up of what follows; once set, it is read without it.
std::mutex g_mu;
std::atomic<int*> g_err_word[kMaxDevices];
std::atomic<int> g_sm_count[kMaxDevices];
std::atomic<uint64_t> g_timeout_ns{0};
std::atomic<int> g_inject_skip_kt{-1};
std::atomic<PFN_cuTensorMapEncodeTiled_v12000> g_encode{nullptr};

int current_device() {
    int d = 0;
    cudaGetDevice(&d);
    return d;
}

void init_device_locked(int d) {
    if (d < 0 || d >= kMaxDevices || g_err_word[d]) return;
    int* w = nullptr;
    // One-time allocation of the 4-byte error word of this device.
    if (cudaMalloc(&w, sizeof(int)) == cudaSuccess) {
        cudaMemset(w, 0, sizeof(int));
        cudaDeviceSynchronize();
    }
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, d);
    g_sm_count[d] = sms > 0 ? sms : 1;
    g_err_word[d] = w;   // last: a set word means that all is set
}
void init_device(int d) {
    if (d < 0 || d >= kMaxDevices || g_err_word[d].load()) return;
    std::lock_guard<std::mutex> lk(g_mu);
    init_device_locked(d);
}
// The tensor-map encoder, looked up once (null if the driver has none).
PFN_cuTensorMapEncodeTiled_v12000 tmap_encoder() {
    PFN_cuTensorMapEncodeTiled_v12000 f = g_encode.load();
    if (f) return f;
    std::lock_guard<std::mutex> lk(g_mu);
    if (!g_encode.load()) {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                             cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess || !fn)
            return nullptr;
        g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    }
    return g_encode.load();
}
}  // namespace

int* device_error_word() {
    const int d = current_device();
    init_device(d);
    return (d >= 0 && d < kMaxDevices) ? g_err_word[d].load() : nullptr;
}

int device_sm_count() {
    const int d = current_device();
    init_device(d);
    return (d >= 0 && d < kMaxDevices) ? g_sm_count[d].load() : 1;
}

uint64_t wait_timeout_ns() {
    uint64_t ns = g_timeout_ns.load();
    if (ns) return ns;
    double ms = 4000.0;   // default: 4 s per wait; no legitimate wait comes close
    if (const char* s = std::getenv("ALP_WAIT_TIMEOUT_MS")) {
        double v = std::atof(s);
        if (v > 0) ms = v;
    }
    // a limit set since the load stays
    const uint64_t first = (uint64_t)(ms * 1e6);
    return g_timeout_ns.compare_exchange_strong(ns, first) ? first : ns;
}

alp_status cuda_status(cudaError_t e) { return e == cudaSuccess ? ALP_OK : ALP_ERR_CUDA; }

alp_status make_tmap_2d(CUtensorMap* map, CUtensorMapDataType dtype, int elem_bytes,
                        const void* base, uint64_t inner, uint64_t outer, uint64_t row_bytes,
                        uint32_t box_inner, uint32_t box_outer, CUtensorMapSwizzle swz) {
    const auto encode = tmap_encoder();
    if (!encode) return ALP_ERR_CUDA;
    (void)elem_bytes;
    cuuint64_t dims[2] = {inner, outer};
    cuuint64_t strides[1] = {row_bytes};
    cuuint32_t box[2] = {box_inner, box_outer};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = encode(map, dtype, 2, const_cast<void*>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? ALP_OK : ALP_ERR_UNSUPPORTED;
}

// 3-D bf16 map (d0 innermost, contiguous rows of d0 elements, d1 rows per
// plane), 128-byte swizzle, box {box0, box1, 1}.
alp_status make_tmap_3d_bf16(CUtensorMap* map, const void* base, uint64_t d0, uint64_t d1,
                             uint64_t d2, uint32_t box0, uint32_t box1) {
    const auto encode = tmap_encoder();
    if (!encode) return ALP_ERR_CUDA;
    cuuint64_t dims[3] = {d0, d1, d2};
    cuuint64_t strides[2] = {d0 * 2, d0 * d1 * 2};
    cuuint32_t box[3] = {box0, box1, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims,
                          strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                          CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? ALP_OK : ALP_ERR_UNSUPPORTED;
}

// The autotuner's pick for 8192^3 on GB300 (0.997 of the measured DMMA peak).
// A call without a config takes it only while the fault-injection hook is on:
// the kernel it otherwise runs (native_direct.cu) has no device-side waits.
static bool default_native_config(alp_config* out) {
    *out = alp_config{64, 128, 64, 4, 4, 0};
    return true;
}

bool default_config(alp_path path, alp_config* out) {
    if (path == ALP_PATH_EMUL) {
        *out = alp_config{256, 256, 64, 2, 0, 16};   // CTA pairs, raster group of 16 tile-rows
        return true;
    }
    return default_native_config(out);
}

int inject_skip_kt() { return g_inject_skip_kt.load(); }

// Shared validation of one GEMM's arguments.
alp_status validate_gemm(int64_t M, int64_t N, int64_t K, double alpha, const void* A,
                         int64_t lda, const void* B, int64_t ldb, double beta, const void* C,
                         int64_t ldc) {
    if (M < 0 || N < 0 || K < 0) return ALP_ERR_INVALID_ARG;
    if (M == 0 || N == 0) return ALP_OK;
    if (lda < K || ldb < N || ldc < N) return ALP_ERR_INVALID_ARG;
    if (!C) return ALP_ERR_INVALID_ARG;
    const bool reads_ab = (alpha != 0.0 && K > 0);
    if (reads_ab && (!A || !B)) return ALP_ERR_INVALID_ARG;
    if (((uintptr_t)C & 7) || (reads_ab && (((uintptr_t)A & 7) || ((uintptr_t)B & 7))))
        return ALP_ERR_INVALID_ARG;   // doubles must be naturally aligned
    (void)beta;
    return ALP_OK;
}

}  // namespace alp

using namespace alp;

extern "C" {

const char* alp_status_string(alp_status s) {
    switch (s) {
        case ALP_OK: return "ALP_OK";
        case ALP_ERR_INVALID_ARG: return "ALP_ERR_INVALID_ARG: invalid argument";
        case ALP_ERR_UNSUPPORTED: return "ALP_ERR_UNSUPPORTED: not supported by this build or input";
        case ALP_ERR_CUDA: return "ALP_ERR_CUDA: a CUDA runtime call failed";
        case ALP_ERR_TIMEOUT: return "ALP_ERR_TIMEOUT: a device-side wait ran past its limit";
        case ALP_ERR_WORKSPACE: return "ALP_ERR_WORKSPACE: workspace missing or too small";
        case ALP_ERR_NOT_TUNED: return "ALP_ERR_NOT_TUNED: no tuned config or cost model";
    }
    return "unknown alp_status";
}

// The tile config of a native call: the caller's, a cached one that was set or
// timed faster than the register-direct kernels, or the default while the
// fault-injection hook is on.  False: none, native_direct runs.
static bool pick_config(int64_t M, int64_t N, int64_t K, const alp_config* cfg, alp_config* c,
                        cudaStream_t s) {
    if (cfg) {
        *c = *cfg;
        return true;
    }
    if (tuned_config(M, N, K, ALP_PATH_NATIVE, c, s)) return true;
    return inject_skip_kt() >= 0 && default_config(ALP_PATH_NATIVE, c);
}

alp_status alp_gemm_f64(int64_t M, int64_t N, int64_t K, double alpha, const double* A,
                        int64_t lda, const double* B, int64_t ldb, double beta, double* C,
                        int64_t ldc, const alp_config* cfg, void* stream) {
    alp_status st = validate_gemm(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc);
    if (st != ALP_OK || M == 0 || N == 0) return st;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (alpha == 0.0 || K == 0) return native_scale(M, N, beta, C, ldc, s);
    alp_config c;
    const bool have = pick_config(M, N, K, cfg, &c, s);
    if (cfg && !native_config_valid(c.bm, c.bn, c.bk, c.tm, c.tn, c.stages))
        return ALP_ERR_INVALID_ARG;
    if (M > 0x7fffffffLL || N > 0x7fffffffLL || K > 0x7fffffffLL) return ALP_ERR_UNSUPPORTED;
    if (!have) return native_direct(0, 0, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, s);
    // TMA wants 16-byte aligned bases and row strides that are multiples of 16 bytes.
    const bool tma_ok = (((uintptr_t)A & 15) == 0) && (((uintptr_t)B & 15) == 0) &&
                        (lda % 2 == 0) && (ldb % 2 == 0);
    return native_launch(c, tma_ok, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, s,
                         inject_skip_kt(), 0);
}

// Bytes of the workspace of alp_gemm_f64_ex: a packed op(A) (M x K) when
// trans_a, then a packed op(B) (K x N) when trans_b, each 256-byte aligned.
static size_t ex_bytes_a(int ta, int64_t M, int64_t K) {
    return ta ? (((size_t)M * (size_t)K * 8 + 255) & ~(size_t)255) : 0;
}
static size_t ex_bytes_b(int tb, int64_t K, int64_t N) {
    return tb ? (((size_t)K * (size_t)N * 8 + 255) & ~(size_t)255) : 0;
}

// Column-major calls: C^T = op(B)^T op(A)^T in row-major terms.
size_t alp_gemm_f64_cm_workspace(int trans_a, int trans_b, int64_t M, int64_t N, int64_t K) {
    return alp_gemm_f64_ex_workspace(trans_b, trans_a, N, M, K);
}

alp_status alp_gemm_f64_cm(int trans_a, int trans_b, int64_t M, int64_t N, int64_t K,
                           double alpha, const double* A, int64_t lda, const double* B,
                           int64_t ldb, double beta, double* C, int64_t ldc,
                           const alp_config* cfg, void* workspace, size_t workspace_bytes,
                           void* stream) {
    return alp_gemm_f64_ex(trans_b, trans_a, N, M, K, alpha, B, ldb, A, lda, beta, C, ldc, cfg,
                           workspace, workspace_bytes, stream);
}

size_t alp_gemm_f64_ex_workspace(int trans_a, int trans_b, int64_t M, int64_t N, int64_t K) {
    if (M < 0 || N < 0 || K < 0 || (trans_a != 0 && trans_a != 1) || (trans_b != 0 && trans_b != 1))
        return 0;
    return ex_bytes_a(trans_a, M, K) + ex_bytes_b(trans_b, K, N);
}

alp_status alp_gemm_f64_ex(int trans_a, int trans_b, int64_t M, int64_t N, int64_t K,
                           double alpha, const double* A, int64_t lda, const double* B,
                           int64_t ldb, double beta, double* C, int64_t ldc,
                           const alp_config* cfg, void* workspace, size_t workspace_bytes,
                           void* stream) {
    if (M < 0 || N < 0 || K < 0 || (trans_a != 0 && trans_a != 1) || (trans_b != 0 && trans_b != 1))
        return ALP_ERR_INVALID_ARG;
    if (!trans_a && !trans_b)
        return alp_gemm_f64(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, cfg, stream);
    if (M == 0 || N == 0) return ALP_OK;
    if (lda < (trans_a ? M : K) || ldb < (trans_b ? K : N) || ldc < N || !C)
        return ALP_ERR_INVALID_ARG;
    const bool reads_ab = alpha != 0.0 && K > 0;
    if (reads_ab && (!A || !B)) return ALP_ERR_INVALID_ARG;
    if (((uintptr_t)C & 7) || (reads_ab && (((uintptr_t)A & 7) || ((uintptr_t)B & 7))))
        return ALP_ERR_INVALID_ARG;
    if (!reads_ab)
        return alp_gemm_f64(M, N, K, alpha, nullptr, K, nullptr, N, beta, C, ldc, cfg, stream);
    const size_t ba = ex_bytes_a(trans_a, M, K), bb = ex_bytes_b(trans_b, K, N);
    if (!workspace || workspace_bytes < ba + bb || ((uintptr_t)workspace & 255))
        return ALP_ERR_WORKSPACE;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    // a pack's grid has at most 65535 x 32 rows of each transposed operand
    if ((trans_a && K > 65535LL * 32) || (trans_b && N > 65535LL * 32)) return ALP_ERR_UNSUPPORTED;
    alp_config c;
    if (!pick_config(M, N, K, cfg, &c, s)) {
        // without a tile config nothing is packed: the operands are read
        // where they are (1021 x 771 x 1333 with A transposed, odd leading
        // dimensions: 3150 us with the pack and the shared-memory kernel,
        // 1960 this way)
        if (M > 0x7fffffffLL || N > 0x7fffffffLL || K > 0x7fffffffLL) return ALP_ERR_UNSUPPORTED;
        return native_direct(trans_a, trans_b, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, s);
    }
    // with one, the transposed operands are packed row-major into the
    // workspace (one read and one write of 8 bytes per element, against 2 M N K
    // flops of FP64 DMMA work), then the product runs as alp_gemm_f64
    char* ws = static_cast<char*>(workspace);
    const double* Aop = A;
    const double* Bop = B;
    int64_t lda_op = lda, ldb_op = ldb;
    alp_status st;
    if (trans_a) {
        double* At = reinterpret_cast<double*>(ws);
        if ((st = native_transpose(A, K, M, lda, At, K, s)) != ALP_OK) return st;
        Aop = At;
        lda_op = K;
    }
    if (trans_b) {
        double* Bt = reinterpret_cast<double*>(ws + ba);
        if ((st = native_transpose(B, N, K, ldb, Bt, N, s)) != ALP_OK) return st;
        Bop = Bt;
        ldb_op = N;
    }
    return alp_gemm_f64(M, N, K, alpha, Aop, lda_op, Bop, ldb_op, beta, C, ldc, cfg, stream);
}

alp_status alp_host_access(int* pageable, int* host_page_tables) {
    if (!pageable || !host_page_tables) return ALP_ERR_INVALID_ARG;
    int d = 0, a = 0, b = 0;
    if (cudaGetDevice(&d) != cudaSuccess ||
        cudaDeviceGetAttribute(&a, cudaDevAttrPageableMemoryAccess, d) != cudaSuccess ||
        cudaDeviceGetAttribute(&b, cudaDevAttrPageableMemoryAccessUsesHostPageTables, d) !=
            cudaSuccess) {
        cudaGetLastError();
        return ALP_ERR_CUDA;
    }
    *pageable = a ? 1 : 0;
    *host_page_tables = b ? 1 : 0;
    return ALP_OK;
}

alp_status alp_get_device_error(void* stream) {
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    int* w = device_error_word();
    if (!w) return ALP_ERR_CUDA;
    int h = 0;
    if (cudaMemcpyAsync(&h, w, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return ALP_ERR_CUDA;
    if (cudaMemsetAsync(w, 0, sizeof(int), s) != cudaSuccess) return ALP_ERR_CUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return ALP_ERR_CUDA;
    return (alp_status)h;
}

// ---- extensions (alp_ext.h) ----

int alp_config_valid(const alp_config* cfg, alp_path path) {
    if (!cfg) return 0;
    if (path == ALP_PATH_NATIVE)
        return native_config_valid(cfg->bm, cfg->bn, cfg->bk, cfg->tm, cfg->tn, cfg->stages) ? 1 : 0;
    if (path == ALP_PATH_EMUL) return emul_config_valid(*cfg) ? 1 : 0;
    return 0;
}

int64_t alp_config_smem_bytes(const alp_config* cfg) {
    if (!cfg) return -1;
    const int s = cfg->stages > 0 ? cfg->stages : native_stages(cfg->bm, cfg->bn, cfg->bk, 0);
    return native_stage_bytes(cfg->bm, cfg->bn, cfg->bk) * s;
}

int alp_config_threads(const alp_config* cfg) {
    if (!cfg) return -1;
    return native_threads(cfg->bm, cfg->bn, cfg->tm, cfg->tn);
}

alp_status alp_set_wait_timeout_ms(double ms) {
    if (!(ms > 0)) return ALP_ERR_INVALID_ARG;
    g_timeout_ns = (uint64_t)(ms * 1e6);
    return ALP_OK;
}

alp_status alp_debug_inject_skip(int kt) {
    g_inject_skip_kt = kt;
    return ALP_OK;
}

}  // extern "C"
