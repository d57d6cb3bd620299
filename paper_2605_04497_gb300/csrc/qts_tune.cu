// Launch-shape autotuner of the forward: times the work per thread block of the
// block-table kernels on the caller's data, keeps the fastest, and optionally
// merges it into a JSON cache keyed by (width, log2 of the work, log2 F, log2 M).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <fstream>
#include <map>
#include <sstream>

#include "qts_blocks.h"

namespace qts {

static int ilog2(int64_t v) {
    int l = 0;
    while (v > 1) { v >>= 1; ++l; }
    return l;
}

// One choice serves the whole ensemble (its buckets share launches); it is kept under the
// width of every path bucket.  `cost`: the estimate of the forward's work per tile.
static std::string cache_key(int D, double cost, int F, int64_t M) {
    return "blocks|" + std::to_string(D) + "|" + std::to_string(ilog2((int64_t)cost)) + "|" +
           std::to_string(ilog2(F)) + "|" + std::to_string(ilog2(std::max<int64_t>(M, 1)));
}

// The cache file is a flat JSON object:
//   {"blocks|D|logCost|logF|logM": [work], ...}
// with Tune::bpaths as `work`.  Entries under other keys (earlier versions kept path
// kernels' parameters under "D|logF|logM") are kept as they are and not used.
static std::map<std::string, std::string> read_cache(const char* path) {
    std::map<std::string, std::string> out;
    std::ifstream in(path);
    if (!in) return out;
    std::stringstream ss;
    ss << in.rdbuf();
    const std::string s = ss.str();
    size_t i = 0;
    while ((i = s.find('"', i)) != std::string::npos) {
        const size_t j = s.find('"', i + 1);
        if (j == std::string::npos) break;
        const size_t lb = s.find('[', j), rb = s.find(']', j);
        if (lb == std::string::npos || rb == std::string::npos || rb < lb) break;
        out[s.substr(i + 1, j - i - 1)] = s.substr(lb + 1, rb - lb - 1);
        i = rb + 1;
    }
    return out;
}

static void write_cache(const char* path, const std::map<std::string, std::string>& m) {
    std::ofstream o(std::string(path) + ".tmp");
    o << "{\n";
    size_t n = 0;
    for (const auto& kv : m) o << "  \"" << kv.first << "\": [" << kv.second << "]" << (++n < m.size() ? "," : "") << "\n";
    o << "}\n";
    o.close();
    std::rename((std::string(path) + ".tmp").c_str(), path);
}

// Tune::bpaths to try; 0, the rule on the call's work, stays unless another is clearly faster
constexpr int kWork[] = {0, 128, 256, 512, 1024, 2048};

// the cached choice under `key`, -1: none that this version writes
static int cached_work(const std::map<std::string, std::string>& cache, const std::string& key) {
    const auto it = cache.find(key);
    if (it == cache.end()) return -1;
    for (int w : kWork)
        if (it->second == std::to_string(w)) return w;
    return -1;
}

template <typename F>
static float time_ms(F&& fn, cudaStream_t st, int reps) {
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    fn();  // warm-up
    std::vector<float> ts;
    for (int r = 0; r < reps; ++r) {
        cudaEventRecord(a, st);
        fn();
        cudaEventRecord(b, st);
        cudaEventSynchronize(b);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, a, b);
        ts.push_back(ms);
    }
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    std::sort(ts.begin(), ts.end());
    return ts[ts.size() / 2];
}

}  // namespace qts

using namespace qts;

extern "C" qts_status qts_autotune(qts_ensemble* e, const float* X, int64_t M, int32_t F,
                                   const char* cache_path, qts_stream_t stream) try {
    qts_status st = check_call(e, X, M, F, 8);
    if (st != QTS_OK) return st;
    if (M == 0) return QTS_OK;
    if (e->flags & QTS_FLAG_FP64) return fail(QTS_ERR_UNSUPPORTED, "autotuning applies to the FP32 kernels");
    cudaStream_t s = (cudaStream_t)stream;
    std::map<std::string, std::string> cache;
    if (cache_path) cache = read_cache(cache_path);
    const int64_t Mt = std::min<int64_t>(M, 4096);  // tune on a leading slice of the samples
    // the FP32 forward runs on the block tables
    st = ensure_blocks(e, false);
    if (st != QTS_OK) return st;
    double cost = 1.0;
    for (const BlockBucket& b : e->blk) cost += (double)b.n * blk_cost(b.D, b.h);
    int best = -1;
    for (const Bucket& b : e->prep.buckets) {
        const int w = cached_work(cache, cache_key(b.D, cost, F, M));
        if (w < 0 || (best >= 0 && w != best)) {
            best = -1;
            break;
        }
        best = w;
    }
    cudaError_t ce = cudaSuccess;
    if (best < 0) {
        double* phi = nullptr;
        ce = cudaMalloc(&phi, sizeof(double) * Mt * (F + 1));
        if (ce != cudaSuccess) {
            cudaGetLastError();
            return cuda_fail(ce, "autotune scratch");
        }
        const int before = e->bpaths;
        float best_ms = 1e30f;
        best = 0;
        for (int work : kWork) {
            e->bpaths = work;
            cudaError_t le = cudaSuccess;
            const float ms = time_ms([&] { le = launch_fwd_blocks(e, X, Mt, F, 8, phi, s); }, s, 5);
            if (le == cudaSuccess && ms < (work == 0 ? 1.f : 0.98f) * best_ms) {
                best_ms = ms;
                best = work;
            }
            cudaGetLastError();
        }
        e->bpaths = before;
        ce = cudaStreamSynchronize(s);
        cudaFree(phi);
        if (ce != cudaSuccess) return cuda_fail(ce, "autotune");
        for (const Bucket& b : e->prep.buckets) cache[cache_key(b.D, cost, F, M)] = std::to_string(best);
    }
    e->bpaths = best;
    ++e->tune_gen;
    batch_forget(e);
    if (cache_path) write_cache(cache_path, cache);
    return QTS_OK;
} QTS_ENTRY_END
