// Autotuner: enumeration of the valid tile configs, CUDA-event timing of each
// on the GPU, the tuned-config cache consulted by the GEMM calls (cfg = NULL),
// and the append-only JSONL timing database.
//
// The paper tunes its tile size T by sweeping powers of two at one matrix
// size (N = 10240, control N = 7168) and keeping the best of ten runs
// (Sect. 2, Sect. 3 "Parameter Tuning", Fig. 3, Table 4).  Here the sweep covers
// the block tile, the K step and the per-thread tile (native path) or the
// raster group (emulated path), for any (M, N, K).
//
// Timing proxy: a large shape would take seconds per config in FP64, so a
// config is timed on one wave of blocks (the first min(tiles, SMs x blocks
// per SM) tiles) with K capped at kProxyK, and the time is scaled by the
// tiles per SM (full problem over proxy: blocks on one SM share its FP64
// pipe) and by K / K'.  Shapes that fit one wave with K <= kProxyK are timed
// exactly.  The emulated path runs its full grid with K capped.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <tuple>
#include <vector>

#include "alp_ext.h"
#include "alp_internal.cuh"
#include "emul.cuh"
#include "native_cfg.h"

namespace alp {

alp_status native_launch(const alp_config& cfg, bool use_tma, int64_t M, int64_t N, int64_t K,
                         double alpha, const double* A, int64_t lda, const double* B,
                         int64_t ldb, double beta, double* C, int64_t ldc, cudaStream_t stream,
                         int inject_skip_kt, int64_t grid_limit);
int native_occupancy(const alp_config& cfg, bool use_tma);
int native_direct_cut(int64_t M, int64_t N, int64_t K, int sms);
alp_status native_direct(int ta, int tb, int64_t M, int64_t N, int64_t K, double alpha,
                         const double* A, int64_t lda, const double* B, int64_t ldb, double beta,
                         double* C, int64_t ldc, cudaStream_t stream, int cut, int64_t tile_limit);
bool default_config(alp_path path, alp_config* out);
bool model_loaded();
bool model_predict(int64_t M, int64_t N, int64_t K, alp_path path, alp_config* out,
                   double* pred_tflops);

namespace {
constexpr int64_t kProxyK = 256;        // K cap of the native timing proxy
// K cap of the emulated timing proxy (env ALP_TUNE_PROXY_K_EMUL, a multiple of
// 64 in [64, 32768]; default 2048).  Measured on GB300 against full-K timings
// of 5 shapes: a cap of 256 over-estimated by 2-3x and ranked the one-block
// kernel above the CTA pairs (wrong by 30 %); 1024 ranked right but
// over-estimated by about 1.3x; 2048 came within 1-12 %.
int64_t proxy_k_emul() {
    if (const char* s = std::getenv("ALP_TUNE_PROXY_K_EMUL")) {
        const long long v = std::atoll(s);
        if (v >= 64 && v <= 32768 && v % 64 == 0) return v;
    }
    return 2048;
}
constexpr int kTimedRuns = 10;          // the paper keeps the best of ten runs

std::mutex g_tmu;
std::atomic<bool> g_cached{false};   // g_cache may have entries
struct Tuned {
    alp_config cfg;
    bool direct;   // timed no faster than the register-direct kernels (native path)
};
std::map<std::tuple<int64_t, int64_t, int64_t, int>, Tuned> g_cache;

const int kBM[3] = {64, 128, 256};
const int kBK[3] = {16, 32, 64};
const int kT[3] = {2, 4, 8};
const int kGroups[6] = {1, 2, 4, 8, 16, 32};

std::vector<alp_config> native_configs() {
    std::vector<alp_config> v;
    for (int bm : kBM)
        for (int bn : kBM)
            for (int bk : kBK)
                for (int tm : kT)
                    for (int tn : kT)
                        if (native_config_valid(bm, bn, bk, tm, tn, 0))
                            v.push_back(alp_config{bm, bn, bk, tm, tn, 0});
    return v;
}

std::vector<alp_config> emul_configs() {
    std::vector<alp_config> v;
    for (int g : kGroups) v.push_back(alp_config{128, 256, 64, 1, 0, g});   // one block
    for (int g : kGroups) v.push_back(alp_config{256, 256, 64, 2, 0, g});   // CTA pairs
    return v;
}

int runs_from_env() {
    if (const char* s = std::getenv("ALP_TUNE_RUNS")) {
        const int v = std::atoi(s);
        if (v >= 1 && v <= 100) return v;
    }
    return kTimedRuns;
}

// Device scratch of one tuning call.
struct Scratch {
    void* p = nullptr;
    size_t bytes = 0;
    ~Scratch() {
        if (p) cudaFree(p);
    }
    bool get(size_t n) {
        if (n <= bytes) return true;
        if (p) cudaFree(p);
        p = nullptr;
        bytes = 0;
        if (cudaMalloc(&p, n) != cudaSuccess) return false;
        bytes = n;
        return cudaMemset(p, 0x3F, n) == cudaSuccess;   // finite, nonzero values
    }
};

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

// Best and median of `runs` event-timed launches (after one warm-up), in ms.
template <class F>
bool time_launch(F&& launch, cudaStream_t st, int runs, double* best, double* median) {
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess) return false;
    if (cudaEventCreate(&e1) != cudaSuccess) return false;
    bool ok = launch() == ALP_OK;
    std::vector<double> t;
    for (int r = 0; ok && r < runs; ++r) {
        cudaEventRecord(e0, st);
        ok = launch() == ALP_OK;
        cudaEventRecord(e1, st);
        if (cudaEventSynchronize(e1) != cudaSuccess) ok = false;
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        t.push_back(ms);
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (!ok || t.empty()) return false;
    std::sort(t.begin(), t.end());
    *best = t.front();
    *median = t[t.size() / 2];
    return true;
}

// Estimated full-problem time (ms) of one config, measured with the proxy
// (or exactly when use_proxy is false or the proxy is the whole problem).
bool time_config(int64_t M, int64_t N, int64_t K, alp_path path, const alp_config& cfg,
                 bool use_proxy, Scratch& sc, cudaStream_t st, int runs, double* est_ms,
                 double* meas_best, double* meas_median) {
    if (path == ALP_PATH_NATIVE) {
        const int64_t Kp = use_proxy ? std::min(K, kProxyK) : K;
        const int64_t tiles = ((M + cfg.bm - 1) / cfg.bm) * ((N + cfg.bn - 1) / cfg.bn);
        // the kernel a call with lda = K, ldb = N would take: TMA needs even
        // leading dimensions (16-byte row strides)
        const bool tma = (K % 2 == 0) && (N % 2 == 0);
        int occ = native_occupancy(cfg, tma);
        if (occ < 1) return false;
        const int64_t slots = (int64_t)device_sm_count() * occ;
        const int64_t run_tiles = use_proxy ? std::min(tiles, slots) : tiles;
        const size_t ba = up256((size_t)M * Kp * 8), bb = up256((size_t)Kp * N * 8);
        const size_t bc = up256((size_t)M * N * 8);
        if (!sc.get(ba + bb + bc)) return false;
        char* base = static_cast<char*>(sc.p);
        const double* A = reinterpret_cast<const double*>(base);
        const double* B = reinterpret_cast<const double*>(base + ba);
        double* C = reinterpret_cast<double*>(base + ba + bb);
        auto launch = [&]() {
            return native_launch(cfg, tma, M, N, Kp, 1.0, A, Kp, B, N, 0.0, C, N, st, -1,
                                 run_tiles);
        };
        if (!time_launch(launch, st, runs, meas_best, meas_median)) return false;
        // co-resident blocks share an SM's FP64 pipe, so time follows the
        // tiles each SM must process: ceil(tiles / SMs) in the full problem
        // against ceil(run_tiles / SMs) in the proxy
        const double sms = (double)device_sm_count();
        const double scale = std::ceil((double)tiles / sms) / std::ceil((double)run_tiles / sms);
        *est_ms = *meas_best * scale * ((double)K / (double)Kp);
        return true;
    }
    // emulated path: the tensor-core stage (its cost dominates), full grid
    const int s = kMaxSlices;
    const int64_t Kp = use_proxy ? std::min(K, proxy_k_emul()) : K;
    const int64_t kpad = (Kp + kEmulBK - 1) / kEmulBK * kEmulBK;
    const int64_t ldg = (N + 255) / 256 * 256;
    const size_t ba = up256((size_t)s * M * kpad * 2), bb = up256((size_t)s * N * kpad * 2);
    const size_t bg = up256((size_t)s * M * ldg * 4);
    if (!sc.get(ba + bb + bg)) return false;
    char* base = static_cast<char*>(sc.p);
    const auto* da = reinterpret_cast<const __nv_bfloat16*>(base);
    const auto* db = reinterpret_cast<const __nv_bfloat16*>(base + ba);
    int32_t* G = reinterpret_cast<int32_t*>(base + ba + bb);
    auto launch = [&]() {
        return emul_slice_gemm(M, N, Kp, s, da, db, kpad, G, ldg, st, cfg.stages,
                               emul_arrangement_of(cfg));
    };
    if (!time_launch(launch, st, runs, meas_best, meas_median)) return false;
    *est_ms = *meas_best * ((double)K / (double)Kp);
    return true;
}

// Estimated time (ms) of the register-direct kernels on the whole problem, as
// the configs' proxy takes it, in the cut the whole problem takes: at most kProxyK
// k per warp (four times that where warps share a k range and exchange their sums,
// which must not count several times over), and kDirectWaves waves of blocks, twice
// as many of clusters, whose last ones end less evenly (629 x 937 x 11136, clusters
// of four: 13.2 ms by 16 waves, 12.8 by 32, 12.7 the call), and more where they are
// shorter than kProxyK k (0.6 ms).  With 16 waves of any length the start and the
// end of the launch counted for all: 232 x 15888 x 80, 20 k per warp, 0.72 ms for
// the 0.61 of the call, and a config of 0.66 was taken instead.
constexpr int64_t kDirectWaves = 16;
bool time_direct(int64_t M, int64_t N, int64_t K, Scratch& sc, cudaStream_t st, int runs,
                 double* est_ms) {
    const int64_t sms = device_sm_count();
    const int cut = native_direct_cut(M, N, K, (int)sms), size = std::max(cut, 1);
    const int64_t tiles = cut ? ((M + 15) / 16) * ((N + 7) / 8) : ((M + 31) / 32) * ((N + 15) / 16);
    const int64_t warps = cut ? 4 * cut : 1;   // that share a k range
    const int64_t Kp = std::min(K, (cut ? 4 : 1) * kProxyK * warps);
    const int64_t least = cut > 1 ? 2 * kDirectWaves : kDirectWaves;
    const int64_t most = std::max(kDirectWaves * kProxyK * warps, least * Kp) * sms / (Kp * size);
    const int64_t run_tiles = std::min(tiles, std::max<int64_t>(most, 1));
    const size_t ba = up256((size_t)M * Kp * 8), bb = up256((size_t)Kp * N * 8);
    if (!sc.get(ba + bb + up256((size_t)M * N * 8))) return false;
    char* base = static_cast<char*>(sc.p);
    const double* A = reinterpret_cast<const double*>(base);
    const double* B = reinterpret_cast<const double*>(base + ba);
    double* C = reinterpret_cast<double*>(base + ba + bb);
    auto launch = [&]() {
        return native_direct(0, 0, M, N, Kp, 1.0, A, Kp, B, N, 0.0, C, N, st, cut, run_tiles);
    };
    double best, median;
    if (!time_launch(launch, st, runs, &best, &median)) return false;
    auto waves = [&](int64_t t) { return std::ceil((double)(t * size) / (double)sms); };
    *est_ms = best * (waves(tiles) / waves(run_tiles)) * ((double)K / (double)Kp);
    return true;
}

void db_append(int64_t M, int64_t N, int64_t K, alp_path path, const std::vector<alp_config>& cs,
               const std::vector<double>& est, const std::vector<double>& best,
               const std::vector<double>& med, int winner, bool proxy, double direct) {
    const char* path_env = std::getenv("ALP_TUNE_DB");
    if (!path_env || !*path_env) return;
    FILE* f = std::fopen(path_env, "a");
    if (!f) return;
    char name[256] = "unknown";
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceProp prop;
    if (cudaGetDeviceProperties(&prop, dev) == cudaSuccess) std::snprintf(name, sizeof name, "%s", prop.name);
    std::string line;
    char buf[512];
    std::snprintf(buf, sizeof buf,
                  "{\"device\": \"%s\", \"M\": %lld, \"N\": %lld, \"K\": %lld, \"path\": \"%s\", "
                  "\"proxy\": %s, \"kcap\": %lld, \"winner\": %d, \"configs\": [",
                  name, (long long)M, (long long)N, (long long)K,
                  path == ALP_PATH_NATIVE ? "native" : "emul", proxy ? "true" : "false",
                  (long long)(path == ALP_PATH_NATIVE ? kProxyK : proxy_k_emul()), winner);
    line += buf;
    for (size_t i = 0; i < cs.size(); ++i) {
        std::snprintf(buf, sizeof buf, "%s[%d, %d, %d, %d, %d, %d, %.6g, %.6g, %.6g]",
                      i ? ", " : "", cs[i].bm, cs[i].bn, cs[i].bk, cs[i].tm, cs[i].tn, cs[i].stages,
                      est[i], best[i], med[i]);
        line += buf;
    }
    line += "]";
    if (std::isfinite(direct)) {   // ms of the register-direct kernels
        std::snprintf(buf, sizeof buf, ", \"direct\": %.6g", direct);
        line += buf;
    }
    line += "}\n";
    std::fputs(line.c_str(), f);
    std::fclose(f);
}

}  // namespace

std::vector<alp_config> configs_of(alp_path path) {
    if (path == ALP_PATH_NATIVE) return native_configs();
    if (path == ALP_PATH_EMUL) return emul_configs();
    return {};
}

void cache_config(int64_t M, int64_t N, int64_t K, alp_path path, const alp_config& c,
                  bool direct = false) {
    std::lock_guard<std::mutex> lk(g_tmu);
    g_cache[std::make_tuple(M, N, K, (int)path)] = {c, direct};
    g_cached.store(true);
}

// Config of a GEMM issued with cfg == NULL: the tuned cache's, else, on the
// emulated path, the cost model's prediction (made once per shape and then
// cached; skipped while `stream` is being captured, since the prediction
// synchronises).  False when there is none, and on the native path also where
// the sweep timed its best config no faster than the register-direct kernels
// (64^3: 73 us with the best config, 6.2 without).  The model, which only knows
// configs, is not asked there: a config's tiles are made of the direct kernels'
// 32 x 16 ones, so its busiest sub-partition never has fewer MMAs (4096^3: 125.1
// ms without a config, 125.6 with the tuned one; 8192 x 8192 x 32, where the ends
// of tiles count most, 4.10 and 4.07).
bool tuned_config(int64_t M, int64_t N, int64_t K, alp_path path, alp_config* out,
                   cudaStream_t stream) {
    if (g_cached.load()) {
        std::lock_guard<std::mutex> lk(g_tmu);
        auto it = g_cache.find(std::make_tuple(M, N, K, (int)path));
        if (it != g_cache.end()) {
            *out = it->second.cfg;
            return !it->second.direct;
        }
    }
    if (path == ALP_PATH_NATIVE) return false;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (model_loaded() && cudaStreamIsCapturing(stream, &cs) == cudaSuccess &&
        cs == cudaStreamCaptureStatusNone &&
        model_predict(M, N, K, path, out, nullptr)) {
        cache_config(M, N, K, path, *out);
        return true;
    }
    cudaGetLastError();
    return false;
}

// The same, with the path's default config where there is no tuned one.
bool select_config(int64_t M, int64_t N, int64_t K, alp_path path, alp_config* out,
                   cudaStream_t stream) {
    return tuned_config(M, N, K, path, out, stream) || default_config(path, out);
}

}  // namespace alp

using namespace alp;

extern "C" {

int alp_config_count(alp_path path) { return (int)configs_of(path).size(); }

alp_status alp_config_at(alp_path path, int idx, alp_config* out) {
    if (!out) return ALP_ERR_INVALID_ARG;
    auto v = configs_of(path);
    if (idx < 0 || idx >= (int)v.size()) return ALP_ERR_INVALID_ARG;
    *out = v[idx];
    return ALP_OK;
}

alp_status alp_tune_time_config(int64_t M, int64_t N, int64_t K, alp_path path,
                                const alp_config* cfg, int use_proxy, int runs,
                                double* est_ms) {
    if (!cfg || !est_ms || M <= 0 || N <= 0 || K <= 0 || runs < 1) return ALP_ERR_INVALID_ARG;
    if (!alp_config_valid(cfg, path)) return ALP_ERR_INVALID_ARG;
    if (path == ALP_PATH_EMUL && K > kEmulMaxK) return ALP_ERR_UNSUPPORTED;
    Scratch sc;
    cudaStream_t st;
    if (cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking) != cudaSuccess) return ALP_ERR_CUDA;
    double b = 0, m = 0;
    const bool ok = time_config(M, N, K, path, *cfg, use_proxy != 0, sc, st, runs, est_ms, &b, &m);
    cudaStreamSynchronize(st);
    cudaStreamDestroy(st);
    return ok ? ALP_OK : ALP_ERR_CUDA;
}

alp_status alp_tune(int64_t M, int64_t N, int64_t K, alp_path path, alp_tune_mode mode,
                    alp_config* out, double* out_tflops) {
    if (!out || M <= 0 || N <= 0 || K <= 0) return ALP_ERR_INVALID_ARG;
    if (path != ALP_PATH_NATIVE && path != ALP_PATH_EMUL) return ALP_ERR_INVALID_ARG;
    const double flops = 2.0 * (double)M * (double)N * (double)K;
    if (mode == ALP_TUNE_LOOKUP) {
        std::lock_guard<std::mutex> lk(g_tmu);
        auto it = g_cache.find(std::make_tuple(M, N, K, (int)path));
        if (it == g_cache.end()) return ALP_ERR_NOT_TUNED;
        *out = it->second.cfg;
        if (out_tflops) *out_tflops = 0.0;
        return ALP_OK;
    }
    if (mode == ALP_TUNE_PREDICT) {
        double tf = 0.0;
        if (!model_predict(M, N, K, path, out, &tf)) return ALP_ERR_NOT_TUNED;
        if (out_tflops) *out_tflops = tf;
        return ALP_OK;
    }
    if (mode != ALP_TUNE_EXHAUSTIVE) return ALP_ERR_INVALID_ARG;
    if (path == ALP_PATH_EMUL && K > kEmulMaxK) return ALP_ERR_UNSUPPORTED;
    const std::vector<alp_config> cs = configs_of(path);
    std::vector<double> est(cs.size(), INFINITY), best(cs.size(), INFINITY), med(cs.size(), INFINITY);
    Scratch sc;
    cudaStream_t st;
    if (cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking) != cudaSuccess) return ALP_ERR_CUDA;
    const int runs = runs_from_env();
    int winner = -1;
    for (size_t i = 0; i < cs.size(); ++i) {
        if (!time_config(M, N, K, path, cs[i], true, sc, st, runs, &est[i], &best[i], &med[i]))
            continue;
        // tie-break: smaller shared memory, then the earlier (lexicographic) config
        if (winner < 0 || est[i] < est[winner] ||
            (est[i] == est[winner] &&
             alp_config_smem_bytes(&cs[i]) < alp_config_smem_bytes(&cs[winner])))
            winner = (int)i;
    }
    double direct = INFINITY;   // a failure leaves the sweep's winner
    if (path == ALP_PATH_NATIVE && !time_direct(M, N, K, sc, st, runs, &direct)) direct = INFINITY;
    cudaStreamSynchronize(st);
    cudaStreamDestroy(st);
    if (winner < 0) return ALP_ERR_CUDA;
    const bool proxy = path == ALP_PATH_NATIVE ? (K > kProxyK) : (K > proxy_k_emul());
    db_append(M, N, K, path, cs, est, best, med, winner, proxy, direct);
    cache_config(M, N, K, path, cs[winner], direct <= est[winner]);
    *out = cs[winner];
    if (out_tflops) *out_tflops = flops / (est[winner] * 1e-3) / 1e12;
    return ALP_OK;
}

alp_status alp_tune_set_cached(int64_t M, int64_t N, int64_t K, alp_path path,
                               const alp_config* cfg) {
    if (!cfg || !alp_config_valid(cfg, path)) return ALP_ERR_INVALID_ARG;
    cache_config(M, N, K, path, *cfg);
    return ALP_OK;
}

alp_status alp_tune_clear_cache(void) {
    std::lock_guard<std::mutex> lk(g_tmu);
    g_cache.clear();
    g_cached.store(false);
    return ALP_OK;
}

}  // extern "C"
