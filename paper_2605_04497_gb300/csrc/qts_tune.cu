// Launch-shape autotuner of the forward: times the work per thread block of the
// block-table kernels on the caller's data, keeps the fastest, and optionally
// merges it into a JSON cache keyed by (width, log2 F, log2 M).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <fstream>
#include <map>
#include <sstream>

#include "qts_internal.h"

namespace qts {

void batch_forget(const qts_ensemble* e);

static int ilog2(int64_t v) {
    int l = 0;
    while (v > 1) { v >>= 1; ++l; }
    return l;
}

static std::string cache_key(int D, int F, int64_t M) {
    return std::to_string(D) + "|" + std::to_string(ilog2(F)) + "|" + std::to_string(ilog2(std::max<int64_t>(M, 1)));
}

// The cache file is a flat JSON object:
//   {"D|logF|logM": [warps, paths, sub, np, bpaths, priv], ...}
static std::map<std::string, Tune> read_cache(const char* path) {
    std::map<std::string, Tune> out;
    std::ifstream in(path);
    if (!in) return out;
    std::stringstream ss;
    ss << in.rdbuf();
    const std::string s = ss.str();
    size_t i = 0;
    while ((i = s.find('"', i)) != std::string::npos) {
        const size_t j = s.find('"', i + 1);
        if (j == std::string::npos) break;
        const std::string key = s.substr(i + 1, j - i - 1);
        const size_t lb = s.find('[', j), rb = s.find(']', j);
        if (lb == std::string::npos || rb == std::string::npos) break;
        int v[6] = {0, 0, 0, 0, 0, 0};
        std::stringstream vs(s.substr(lb + 1, rb - lb - 1));
        std::string tok;
        int k = 0;
        while (k < 6 && std::getline(vs, tok, ',')) v[k++] = std::atoi(tok.c_str());
        if (k == 6) out[key] = Tune{v[0], v[1], v[2], v[3], v[4], v[5]};
        i = rb + 1;
    }
    return out;
}

static void write_cache(const char* path, const std::map<std::string, Tune>& m) {
    std::ofstream o(std::string(path) + ".tmp");
    o << "{\n";
    size_t n = 0;
    for (const auto& kv : m) {
        const Tune& t = kv.second;
        o << "  \"" << kv.first << "\": [" << t.warps << ", " << t.paths << ", " << t.sub << ", " << t.np
          << ", " << t.bpaths << ", " << t.priv << "]" << (++n < m.size() ? "," : "") << "\n";
    }
    o << "}\n";
    o.close();
    std::rename((std::string(path) + ".tmp").c_str(), path);
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
    std::map<std::string, Tune> cache;
    if (cache_path) cache = read_cache(cache_path);
    const int64_t Mt = std::min<int64_t>(M, 4096);  // tune on a leading slice of the samples
    double* phi = nullptr;
    // the FP32 forward runs on the block tables
    st = ensure_blocks(e, false);
    if (st != QTS_OK) return st;
    cudaError_t ce = cudaMalloc(&phi, sizeof(double) * Mt * (F + 1));
    if (ce != cudaSuccess) return cuda_fail(ce, "autotune scratch");
    // one choice for the ensemble (its buckets share launches), kept under the
    // width of every path bucket: Tune::bpaths
    bool cached = !e->prep.buckets.empty();
    for (const Bucket& b : e->prep.buckets) cached = cached && cache.count(cache_key(b.D, F, M)) != 0;
    Tune best = e->tune[0];
    if (cached) {
        best = cache[cache_key(e->prep.buckets.front().D, F, M)];
    } else {
        float best_ms = 1e30f;
        for (int paths : {128, 256, 512, 1024, 2048}) {
            for (Tune& t : e->tune) t.bpaths = paths;
            cudaError_t le = cudaSuccess;
            const float ms = time_ms([&] { le = launch_fwd_blocks(e, X, Mt, F, 8, phi, s); }, s, 3);
            if (le == cudaSuccess && ms < best_ms) {
                best_ms = ms;
                best.bpaths = paths;
            }
            cudaGetLastError();
        }
        for (const Bucket& b : e->prep.buckets) cache[cache_key(b.D, F, M)] = best;
    }
    for (Tune& t : e->tune) t.bpaths = best.bpaths;
    ce = cudaStreamSynchronize(s);
    cudaFree(phi);
    if (ce != cudaSuccess) return cuda_fail(ce, "autotune");
    e->tuned = true;
    ++e->tune_gen;
    batch_forget(e);
    if (cache_path) write_cache(cache_path, cache);
    return QTS_OK;
} QTS_ENTRY_END
