// C-ABI entry points: handle lifecycle, argument checks, per-bucket launches.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <memory>
#include <mutex>
#include <new>

#include "qts_device.cuh"
#include "qts_internal.h"

namespace qts {

static thread_local std::string g_err = "no error";

void set_error(const std::string& msg) { g_err = msg; }

qts_status fail(qts_status st, const std::string& msg) {
    g_err = msg;
    return st;
}

qts_status cuda_fail(cudaError_t e, const char* what) {
    g_err = std::string(what) + ": " + cudaGetErrorName(e) + " (" + cudaGetErrorString(e) + ")";
    return e == cudaErrorMemoryAllocation ? QTS_ERR_OOM : QTS_ERR_CUDA;
}

int num_sms() {
    static int sms = 0;
    static std::once_flag once;
    std::call_once(once, [] {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            sms = 152;
    });
    return sms;
}

static Tune default_tune(int D) {
    Tune t;
    t.warps = 4;
    t.sub = D <= 16 ? 32 : 16;
    t.paths = D <= 8 ? 512 : (D <= 16 ? 256 : 128);
    return t;
}

void release_device(qts_ensemble* e) {
    cudaFree(e->d_rec);
    cudaFree(e->d_path_leaf);
    cudaFree(e->d_path_zprod);
    cudaFree(e->d_path_val);
    cudaFree(e->d_slot_zexcl);
    cudaFree(e->d_slot_edge_begin);
    cudaFree(e->d_edge_node);
    cudaFree(e->d_edge_coef);
    cudaFree(e->d_empty_leaf);
    e->d_rec = nullptr;
    e->d_path_leaf = nullptr;
    e->d_path_zprod = nullptr;
    e->d_path_val = nullptr;
    e->d_slot_zexcl = nullptr;
    e->d_slot_edge_begin = nullptr;
    e->d_edge_node = nullptr;
    e->d_edge_coef = nullptr;
    e->d_empty_leaf = nullptr;
    e->device_bytes = 0;
    release_dfs(e);
    cudaFree(e->d_pair_rec);
    e->d_pair_rec = nullptr;
    e->pair_ready = false;
    release_blocks(e);
}

template <typename T>
static qts_status up(T** dst, const std::vector<T>& src, int64_t* total, const char* what) {
    size_t bytes = std::max<size_t>(src.size(), 1) * sizeof(T);
    cudaError_t err = cudaMalloc((void**)dst, bytes);
    if (err != cudaSuccess) return cuda_fail(err, what);
    if (!src.empty()) {
        err = cudaMemcpy(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice);
        if (err != cudaSuccess) return cuda_fail(err, what);
    }
    *total += (int64_t)bytes;
    return QTS_OK;
}

qts_status upload(qts_ensemble* e) {
    const Prepared& P = e->prep;
    int64_t tot = 0;
    qts_status st = QTS_OK;
    if (e->flags & QTS_FLAG_FP64) st = up((Rec64**)&e->d_rec, P.rec64, &tot, "upload path tables");
    else st = up((Rec32**)&e->d_rec, P.rec32, &tot, "upload path tables");
    if (st == QTS_OK) st = up(&e->d_path_leaf, P.path_leaf, &tot, "upload path leaves");
    if (st == QTS_OK) st = up(&e->d_path_zprod, P.path_zprod, &tot, "upload path products");
    if (st == QTS_OK) st = up(&e->d_path_val, P.path_val, &tot, "upload path values");
    if (st == QTS_OK) st = up(&e->d_slot_zexcl, P.slot_zexcl, &tot, "upload element products");
    if (st == QTS_OK) st = up(&e->d_slot_edge_begin, P.slot_edge_begin, &tot, "upload element edges");
    if (st == QTS_OK) st = up(&e->d_edge_node, P.edge_node, &tot, "upload edge nodes");
    if (st == QTS_OK) st = up(&e->d_edge_coef, P.edge_coef, &tot, "upload edge coefficients");
    if (st == QTS_OK) st = up(&e->d_empty_leaf, P.empty_leaf, &tot, "upload single-leaf trees");
    if (st != QTS_OK) {
        release_device(e);
        return st;
    }
    e->device_bytes = tot;
    // the device copies are the working set; keep only sizes and bucket info
    Prepared& Pm = e->prep;
    std::vector<Rec32>().swap(Pm.rec32);
    std::vector<Rec64>().swap(Pm.rec64);
    std::vector<int64_t>().swap(Pm.path_leaf);
    std::vector<double>().swap(Pm.path_zprod);
    std::vector<double>().swap(Pm.path_val);
    std::vector<double>().swap(Pm.slot_zexcl);
    std::vector<int64_t>().swap(Pm.slot_edge_begin);
    std::vector<int64_t>().swap(Pm.edge_node);
    std::vector<double>().swap(Pm.edge_coef);
    return QTS_OK;
}

static void free_blocks(BlockDev& T) {
    for (void* p : {(void*)T.rec, (void*)T.dbl, (void*)T.ent, (void*)T.bias_leaf, (void*)T.bias_z}) cudaFree(p);
    T = BlockDev();
}

// Allocations and copies of tables that a call builds on first use.  The call may be
// under stream capture, on this thread or another, where cudaMalloc is refused
// unless the thread's capture mode is relaxed and a copy on the legacy stream
// would break the capture; so the copies go through a stream of their own, and the
// tables are there when the call returns, whatever becomes of the graph.
struct TableUpload {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaStream_t st = nullptr;
    cudaError_t err;
    TableUpload() {
        err = cudaThreadExchangeStreamCaptureMode(&mode);
        if (err == cudaSuccess) err = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
    }
    ~TableUpload() {
        if (st) cudaStreamDestroy(st);
        cudaThreadExchangeStreamCaptureMode(&mode);
    }
    TableUpload(const TableUpload&) = delete;
    TableUpload& operator=(const TableUpload&) = delete;
    template <typename T>
    void add(T** dst, const std::vector<T>& src) {
        const size_t bytes = std::max<size_t>(src.size(), 1) * sizeof(T);
        if (err == cudaSuccess) err = cudaMalloc((void**)dst, bytes);
        if (err == cudaSuccess && !src.empty())
            err = cudaMemcpyAsync(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice, st);
    }
    cudaError_t finish() {
        if (err == cudaSuccess) err = cudaStreamSynchronize(st);
        return err;
    }
};

// The path tables with sibling leaves merged: prepared from the host copy of the model;
// on the host only their counts are kept.
qts_status ensure_pairs(qts_ensemble* e, bool records) {
    std::lock_guard<std::mutex> lk(e->blk_mu);
    if (e->pair_ready && (!records || e->d_pair_rec)) return QTS_OK;
    Prepared P;
    std::string err;
    const bool cat = !e->is_cat.empty();
    qts_status st = prepare(e->n_trees, e->off.data(), e->left.data(), e->right.data(), e->feature.data(),
                            e->thr.data(), e->defl.data(), e->z.data(), e->leaf.data(),
                            cat ? e->is_cat.data() : nullptr, cat ? e->cat_left.data() : nullptr,
                            e->n_features, false, &P, &err, true);
    if (st != QTS_OK) return fail(st, err);
    if (records) {
        Rec32* rec = nullptr;
        TableUpload up;
        up.add(&rec, P.rec32);
        const cudaError_t ce = up.finish();
        if (ce != cudaSuccess) {
            if (ce == cudaErrorMemoryAllocation) cudaGetLastError();
            cudaFree(rec);
            return cuda_fail(ce, "upload pair tables");
        }
        e->d_pair_rec = rec;
    }
    if (!e->pair_ready) {
        e->pair_sizes.buckets = P.buckets;
        e->pair_sizes.n_paths = P.n_paths;
        e->pair_sizes.sum_unique = P.sum_unique;
        e->pair_sizes.n_pair_paths = P.n_pair_paths;
        e->pair_ready = true;
    }
    return QTS_OK;
}

// Block tables: built from the host copy of the model; `grad` adds the adjoint's
// part.  The records are the same either way: once they are there nothing that a
// forward on another thread or a captured graph uses changes, also on failure.
qts_status ensure_blocks(qts_ensemble* e, bool grad) {
    std::lock_guard<std::mutex> lk(e->blk_mu);
    if (e->blk_ready && (!grad || e->blk_grad_ready)) return QTS_OK;
    grad = grad || e->wants_grad;  // (!blk_ready: a refit step's forward comes first)
    e->wants_grad = grad;
    if (grad && e->n_nodes >= ((int64_t)1 << 31)) return fail(QTS_ERR_UNSUPPORTED, "gradients of 2^31 nodes or more");
    BlockHost H;
    build_blocks(e, grad, &H);
    if (grad && H.n_slots >= ((int64_t)1 << 32)) return fail(QTS_ERR_UNSUPPORTED, "too many adjoint sums");
    BlockDev T;
    TableUpload up;
    if (!e->blk_ready) {
        up.add(&T.rec, H.rec);
        if (!H.dbl.empty()) up.add(&T.dbl, H.dbl);
    }
    if (grad) {
        up.add(&T.ent, H.ent);
        up.add(&T.bias_leaf, H.bias_leaf);
        up.add(&T.bias_z, H.bias_z);
    }
    const cudaError_t err = up.finish();
    if (err != cudaSuccess) {
        if (err == cudaErrorMemoryAllocation) cudaGetLastError();
        free_blocks(T);
        return cuda_fail(err, "upload block tables");
    }
    if (!e->blk_ready) {
        e->blkdev.rec = T.rec;
        e->blkdev.dbl = T.dbl;
        e->blk = std::move(H.buckets);
        e->n_blocks = H.n_blocks;
        e->n_blk_slots = H.n_slots;
        e->blk_ready = true;
    }
    if (grad) {
        e->blkdev.ent = T.ent;
        e->blkdev.n_ent = (int64_t)H.ent.size();
        e->blkdev.bias_leaf = T.bias_leaf;
        e->blkdev.bias_z = T.bias_z;
        e->blk_grad_ready = true;
    }
    return QTS_OK;
}

void release_blocks(qts_ensemble* e) {
    free_blocks(e->blkdev);
    e->blk.clear();
    e->n_blocks = e->n_blk_slots = 0;
    e->blk_ready = e->blk_grad_ready = false;
}

bool is_capturing(cudaStream_t st) {
    cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &s) != cudaSuccess) {
        cudaGetLastError();  // the legacy stream, while another stream is being captured
        return false;
    }
    return s == cudaStreamCaptureStatusActive;
}

// A captured call leaves the workspace's address in the caller's graph, which may be
// replayed after any later call: such a workspace is never freed before the
// ensemble, a call that outgrows it gets a new one beside it.
qts_status ensure_workspace_uncaptured(qts_ensemble* e, size_t bytes) {
    if (bytes > e->work_bytes) {
        if (e->d_work) {
            batch_forget(e);
            cudaError_t err = cudaDeviceSynchronize();
            if (err != cudaSuccess) return cuda_fail(err, "workspace resize sync");
            if (e->work_captured) e->retired.push_back(e->d_work);
            else cudaFree(e->d_work);
            e->d_work = nullptr;
            e->work_bytes = 0;
            e->work_captured = false;
        }
        size_t want = std::max(bytes, (size_t)1 << 20);
        cudaError_t err = cudaMalloc(&e->d_work, want);
        if (err != cudaSuccess) {
            e->d_work = nullptr;
            cudaGetLastError();  // not the next launch's error
            return cuda_fail(err, "workspace allocation");
        }
        e->work_bytes = want;
    }
    return QTS_OK;
}

qts_status ensure_workspace(qts_ensemble* e, size_t bytes, cudaStream_t st) {
    const qts_status r = ensure_workspace_uncaptured(e, bytes);
    if (r == QTS_OK && !e->work_captured && is_capturing(st)) e->work_captured = true;
    return r;
}

// The device failure path on demand: one block waits, bounded, on an mbarrier
// that nothing arrives at; the wait runs out and latches QTS_ERR_TIMEOUT in the
// status word.  No copy is issued, so nothing is left in flight.
__global__ void wait_selftest_kernel(int* status) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_fence_init();
    }
    __syncthreads();
    if (threadIdx.x == 0 && !mbar_wait_bounded(&bar, 0)) report(status, QTS_ERR_TIMEOUT);
}

cudaError_t launch_wait_selftest(int* status, cudaStream_t st) {
    wait_selftest_kernel<<<1, 32, 0, st>>>(status);
    return cudaGetLastError();
}

qts_status check_call(qts_ensemble* e, const float* X, int64_t M, int32_t F, int32_t n_quad) {
    if (!e) return fail(QTS_ERR_ARG, "ensemble handle is NULL");
    if (F != e->n_features)
        return fail(QTS_ERR_ARG, "F = " + std::to_string(F) + " does not match the ensemble's " +
                                     std::to_string(e->n_features) + " features");
    if (M < 0) return fail(QTS_ERR_ARG, "M must be >= 0");
    if (M > 0 && !X) return fail(QTS_ERR_ARG, "X is NULL");
    if (M > ((int64_t)1 << 31)) return fail(QTS_ERR_UNSUPPORTED, "M above 2^31 samples");
    if (n_quad != QTS_NQ_EXACT && (n_quad < 1 || n_quad > QTS_MAX_QUAD))
        return fail(QTS_ERR_ARG, "n_quad must be QTS_NQ_EXACT or in [1, " + std::to_string(QTS_MAX_QUAD) + "]");
    return QTS_OK;
}

}  // namespace qts

using namespace qts;

extern "C" {

const char* qts_last_error(void) { return g_err.c_str(); }

qts_status qts_gauss_legendre(int32_t n, double* t, double* w) {
    if (!t || !w || n < 1 || n > 64) return fail(QTS_ERR_ARG, "n must be in [1, 64] and t, w non-NULL");
    return gauss_legendre(n, t, w) ? QTS_OK : fail(QTS_ERR_ARG, "gauss_legendre failed");
}

int32_t qts_exact_nodes(int32_t width, int32_t order) {
    if (width < 1 || width > QTS_MAX_UNIQUE_FEATURES_PER_PATH || order < 1) return 0;
    return exact_nodes(width, order);
}

static qts_status load_impl(int32_t n_trees, const int64_t* off, const int32_t* left,
                            const int32_t* right, const int32_t* feature, const float* threshold,
                            const uint8_t* default_left, const float* z, const float* leaf_value,
                            const uint8_t* is_cat, const uint64_t* cat_left, int32_t n_features,
                            uint32_t flags, qts_ensemble** out) try {
    if (!out) return fail(QTS_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (n_trees < 1 || !off || !left || !right || !feature || !threshold || !z || !leaf_value)
        return fail(QTS_ERR_ARG, "n_trees < 1 or a required array is NULL");
    if (n_features < 1 || n_features > QTS_MAX_FEATURES)
        return fail(QTS_ERR_UNSUPPORTED, "n_features must be in [1, " + std::to_string(QTS_MAX_FEATURES) + "]");
    if (flags & ~QTS_FLAG_FP64) return fail(QTS_ERR_ARG, "unknown flags");
    if (is_cat && !cat_left) return fail(QTS_ERR_ARG, "category_left_mask is NULL");
    for (int t = 0; t < n_trees; ++t)
        if (off[t + 1] <= off[t]) return fail(QTS_ERR_ARG, "tree_node_offsets must be increasing");
    if (off[0] != 0) return fail(QTS_ERR_ARG, "tree_node_offsets[0] must be 0");
    struct Drop {  // an error on the way, thrown or returned, leaves nothing behind
        void operator()(qts_ensemble* p) const {
            release_device(p);
            cudaFree(p->d_status);
            delete p;
        }
    };
    std::unique_ptr<qts_ensemble, Drop> e(new qts_ensemble());
    const int64_t N = off[n_trees];
    e->n_trees = n_trees;
    e->n_features = n_features;
    e->n_nodes = N;
    e->flags = flags;
    cudaGetDevice(&e->device);
    e->off.assign(off, off + n_trees + 1);
    e->left.assign(left, left + N);
    e->right.assign(right, right + N);
    e->feature.assign(feature, feature + N);
    e->thr.assign(threshold, threshold + N);
    e->z.assign(z, z + N);
    e->leaf.assign(leaf_value, leaf_value + N);
    if (default_left) e->defl.assign(default_left, default_left + N);
    else e->defl.assign((size_t)N, 1);
    if (is_cat) {
        e->is_cat.assign(is_cat, is_cat + N);
        e->cat_left.assign(cat_left, cat_left + N);
    }
    std::string err;
    qts_status st = prepare(n_trees, e->off.data(), e->left.data(), e->right.data(),
                            e->feature.data(), e->thr.data(), e->defl.data(), e->z.data(),
                            e->leaf.data(), is_cat ? e->is_cat.data() : nullptr,
                            is_cat ? e->cat_left.data() : nullptr, n_features,
                            (flags & QTS_FLAG_FP64) != 0, &e->prep, &err);
    if (st != QTS_OK) return fail(st, err);
    cudaError_t ce = cudaMalloc(&e->d_status, sizeof(int));
    if (ce == cudaSuccess) ce = cudaMemset(e->d_status, 0, sizeof(int));
    if (ce != cudaSuccess) return cuda_fail(ce, "status word");
    st = upload(e.get());
    if (st != QTS_OK) return st;
    for (int D = 0; D <= kMaxD; ++D) e->tune[D] = default_tune(std::max(D, 1));
    *out = e.release();
    return QTS_OK;
} QTS_ENTRY_END

qts_status qts_load_ensemble(int32_t n_trees, const int64_t* off, const int32_t* left,
                             const int32_t* right, const int32_t* feature, const float* threshold,
                             const uint8_t* default_left, const float* z, const float* leaf_value,
                             int32_t n_features, uint32_t flags, qts_ensemble** out) {
    return load_impl(n_trees, off, left, right, feature, threshold, default_left, z, leaf_value,
                     nullptr, nullptr, n_features, flags, out);
}

qts_status qts_load_ensemble_cat(int32_t n_trees, const int64_t* off, const int32_t* left,
                                 const int32_t* right, const int32_t* feature, const float* threshold,
                                 const uint8_t* default_left, const float* z, const float* leaf_value,
                                 const uint8_t* is_categorical, const uint64_t* category_left_mask,
                                 int32_t n_features, uint32_t flags, qts_ensemble** out) {
    return load_impl(n_trees, off, left, right, feature, threshold, default_left, z, leaf_value,
                     is_categorical, category_left_mask, n_features, flags, out);
}

qts_status qts_update_params(qts_ensemble* e, const float* z, const float* leaf_value) try {
    if (!e || !z || !leaf_value) return fail(QTS_ERR_ARG, "NULL argument");
    Prepared P;
    std::string err;
    const bool cat = !e->is_cat.empty();
    qts_status st = prepare(e->n_trees, e->off.data(), e->left.data(), e->right.data(),
                            e->feature.data(), e->thr.data(), e->defl.data(), z, leaf_value,
                            cat ? e->is_cat.data() : nullptr,
                            cat ? e->cat_left.data() : nullptr, e->n_features,
                            (e->flags & QTS_FLAG_FP64) != 0, &P, &err);
    if (st != QTS_OK) return fail(st, err);
    cudaError_t ce = cudaDeviceSynchronize();
    if (ce != cudaSuccess) return cuda_fail(ce, "update sync");
    batch_forget(e);
    release_device(e);
    e->z.assign(z, z + e->n_nodes);  // no new memory: the sizes are the same
    e->leaf.assign(leaf_value, leaf_value + e->n_nodes);
    e->prep = std::move(P);
    return upload(e);
} QTS_ENTRY_END

qts_status qts_shap_values(qts_ensemble* e, const float* X, int64_t M, int32_t F, int32_t n_quad,
                           double* phi, qts_stream_t stream) try {
    qts_status st = check_call(e, X, M, F, n_quad);
    if (st != QTS_OK) return st;
    if (M == 0) return QTS_OK;
    if (!phi) return fail(QTS_ERR_ARG, "phi is NULL");
    cudaStream_t s = (cudaStream_t)stream;
    // the block tables (built on the first call that needs them)
    st = ensure_blocks(e, false);
    if (st != QTS_OK) return st;
    cudaError_t ce = launch_phi_init(phi, M, F, e->prep.bias, s);
    if (ce != cudaSuccess) return cuda_fail(ce, "phi init launch");
    if (e->flags & QTS_FLAG_FP64) ce = launch_fwd64(e, X, M, F, n_quad, phi, s);
    else if (M <= kFewRows) ce = launch_fwd_few(e, X, M, F, n_quad, phi, s);
    else ce = launch_fwd_blocks(e, X, M, F, n_quad, phi, s);
    return ce == cudaSuccess ? QTS_OK : cuda_fail(ce, "forward kernel launch");
} QTS_ENTRY_END

qts_status qts_selftest_wait_timeout(qts_ensemble* e, qts_stream_t stream) {
    if (!e) return fail(QTS_ERR_ARG, "ensemble handle is NULL");
    cudaError_t ce = launch_wait_selftest(e->d_status, (cudaStream_t)stream);
    if (ce != cudaSuccess) return cuda_fail(ce, "self-test launch");
    return QTS_OK;
}

qts_status qts_sync_status(qts_ensemble* e, qts_stream_t stream) {
    if (!e) return fail(QTS_ERR_ARG, "ensemble handle is NULL");
    cudaError_t ce = cudaStreamSynchronize((cudaStream_t)stream);
    if (ce != cudaSuccess) return cuda_fail(ce, "stream synchronize");
    int h = 0;
    ce = cudaMemcpy(&h, e->d_status, sizeof(int), cudaMemcpyDeviceToHost);
    if (ce != cudaSuccess) return cuda_fail(ce, "status read");
    if (h != 0) {
        cudaMemset(e->d_status, 0, sizeof(int));
        return fail((qts_status)h, h == QTS_ERR_TIMEOUT ? "a bounded device wait ran out"
                                                        : "device-side check failed");
    }
    return QTS_OK;
}

qts_status qts_get_info(const qts_ensemble* e, qts_info* out) {
    if (!e || !out) return fail(QTS_ERR_ARG, "NULL argument");
    std::memset(out, 0, sizeof(*out));
    out->n_trees = e->n_trees;
    out->n_features = e->n_features;
    out->n_nodes = e->n_nodes;
    out->n_leaves = e->prep.n_leaves;
    out->n_paths = e->prep.n_paths;
    out->max_unique = e->prep.max_unique;
    out->sum_unique = e->prep.sum_unique;
    out->n_buckets = (int32_t)e->prep.buckets.size();
    for (size_t i = 0; i < e->prep.buckets.size() && i < 32; ++i) {
        out->bucket_width[i] = e->prep.buckets[i].D;
        out->bucket_paths[i] = e->prep.buckets[i].n_paths;
    }
    out->expected_value = e->prep.bias;
    out->device_bytes = e->device_bytes;
    out->flags = e->flags;
    return QTS_OK;
}

qts_status qts_describe_ensemble(int32_t n_trees, const int64_t* off, const int32_t* left,
                                 const int32_t* right, const int32_t* feature, const float* threshold,
                                 const uint8_t* default_left, const float* z, const float* leaf_value,
                                 int32_t n_features, uint32_t flags, qts_info* out) try {
    if (!out || n_trees < 1 || !off || !left || !right || !feature || !threshold || !z || !leaf_value)
        return fail(QTS_ERR_ARG, "NULL argument or n_trees < 1");
    if (n_features < 1 || n_features > QTS_MAX_FEATURES)
        return fail(QTS_ERR_UNSUPPORTED, "n_features out of range");
    for (int t = 0; t < n_trees; ++t)
        if (off[t + 1] <= off[t]) return fail(QTS_ERR_ARG, "tree_node_offsets must be increasing");
    std::vector<uint8_t> defl;
    if (!default_left) defl.assign((size_t)off[n_trees], 1);
    Prepared P;
    std::string err;
    const bool fp64 = (flags & QTS_FLAG_FP64) != 0;
    const bool pairs = (flags & QTS_DESCRIBE_PAIRS) != 0;
    qts_status st = prepare(n_trees, off, left, right, feature, threshold,
                            default_left ? default_left : defl.data(), z, leaf_value, nullptr, nullptr,
                            n_features, fp64, &P, &err, pairs);
    if (st != QTS_OK) return fail(st, err);
    std::memset(out, 0, sizeof(*out));
    out->n_trees = n_trees;
    out->n_features = n_features;
    out->n_nodes = off[n_trees];
    out->n_leaves = P.n_leaves;
    out->n_paths = P.n_paths;
    out->max_unique = P.max_unique;
    out->sum_unique = P.sum_unique;
    out->n_buckets = (int32_t)P.buckets.size();
    for (size_t i = 0; i < P.buckets.size() && i < 32; ++i) {
        out->bucket_width[i] = P.buckets[i].D;
        out->bucket_paths[i] = P.buckets[i].n_paths;
    }
    out->expected_value = P.bias;
    out->device_bytes = (int64_t)((fp64 ? P.rec64.size() * sizeof(Rec64) : P.rec32.size() * sizeof(Rec32)) +
                                  P.path_leaf.size() * 8 + P.path_zprod.size() * 8 +
                                  P.slot_edge_begin.size() * 8 + P.edge_node.size() * 16);
    out->flags = flags;
    return QTS_OK;
} QTS_ENTRY_END

qts_status qts_describe_paths(int32_t n_trees, const int64_t* off, const int32_t* left, const int32_t* right,
                              const int32_t* feature, const float* threshold, const uint8_t* default_left,
                              const float* z, const float* leaf_value, const uint8_t* is_categorical,
                              const uint64_t* category_left_mask, int32_t n_features, int64_t* n_records,
                              int64_t* n_paths, uint32_t* records, int64_t* path_leaf, int32_t* path_width) try {
    if (!n_records || !n_paths || n_trees < 1 || !off || !left || !right || !feature || !threshold || !z ||
        !leaf_value)
        return fail(QTS_ERR_ARG, "NULL argument or n_trees < 1");
    if (n_features < 1 || n_features > QTS_MAX_FEATURES)
        return fail(QTS_ERR_UNSUPPORTED, "n_features out of range");
    if (is_categorical && !category_left_mask) return fail(QTS_ERR_ARG, "category_left_mask is NULL");
    for (int t = 0; t < n_trees; ++t)
        if (off[t + 1] <= off[t]) return fail(QTS_ERR_ARG, "tree_node_offsets must be increasing");
    std::vector<uint8_t> defl;
    if (!default_left) defl.assign((size_t)off[n_trees], 1);
    Prepared P;
    std::string err;
    qts_status st = prepare(n_trees, off, left, right, feature, threshold,
                            default_left ? default_left : defl.data(), z, leaf_value, is_categorical,
                            category_left_mask, n_features, false, &P, &err);
    if (st != QTS_OK) return fail(st, err);
    *n_records = (int64_t)P.rec32.size();
    *n_paths = P.n_paths;
    if (!records) return QTS_OK;
    if (!path_leaf || !path_width) return fail(QTS_ERR_ARG, "path_leaf or path_width is NULL");
    std::memcpy(records, P.rec32.data(), P.rec32.size() * sizeof(Rec32));
    std::memcpy(path_leaf, P.path_leaf.data(), P.path_leaf.size() * sizeof(int64_t));
    for (const Bucket& b : P.buckets)
        for (int64_t p = 0; p < b.n_paths; ++p) path_width[b.path_base + p] = b.D;
    return QTS_OK;
} QTS_ENTRY_END

void qts_free(qts_ensemble* e) {
    if (!e) return;
    batch_forget(e);
    cudaDeviceSynchronize();
    release_device(e);
    cudaFree(e->d_status);
    cudaFree(e->d_work);
    for (void* p : e->retired) cudaFree(p);
    delete e;
}

}  // extern "C"
