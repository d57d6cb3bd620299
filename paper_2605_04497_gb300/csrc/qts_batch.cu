// Batched forward + adjoint of many heterogeneous requests in one persistent
// kernel per register class, captured (with its initialisation and epilogues)
// into a CUDA graph; a single adjoint call launches the same kernels.
//
// Work items are (request, bucket, run of blocks, sample tile).  Items are not
// materialised: segments (request, bucket) are ordered by per-item cost,
// heaviest first, and carry their first item index, so a thread block that takes
// item k from the atomic counter finds its segment by binary search.  For a
// request with grad_phi one pass over each (sample, block) yields both phi and
// the adjoint sums (the forward products are part of the adjoint's).
//
// Bound by instruction issue and FP32 (8 to 16 warps per SM).  Measured, path
// tables before and block tables now: eight requests of 17-100 trees, depth 4-13,
// 40-2,000 samples 8.61 -> 4.60 ms (4.10 with the classes' kernels as parallel
// branches); sixteen of at most 200 samples 3.28 -> 0.38 ms (0.15 with one launch for
// all requests' preparation and epilogue; by
// default the warps of a thread block now share 64 samples and split the blocks:
// with 64 samples per warp a request of fewer than 193 left warps idle); adjoint
// alone, 200 trees of depth 8, 4,001 samples 3.30 -> 1.93 ms.
//
// qts-build-parts: 12 (part 0: host code; parts 1-3: the pass of two samples per
// lane, parts 4-11: the others, one register class each)
#include <algorithm>
#include <cstring>
#include <mutex>
#include <numeric>

#include "qts_blocks.cuh"

namespace qts {

struct SegDev {
    const Rec32* rec;
    double* g;          // the bucket's adjoint sums (nullptr: forward only)
    int64_t n;          // blocks
    int64_t item_begin;
    int32_t D, h;
    int32_t per_item;   // blocks per item
    int32_t n_tiles;    // sample groups per run of blocks
    int32_t req;
    int32_t mode;       // 0: the warps share 32 samples and a phi tile (atomics) - forward
                        // only, or too many features for the others; 2: each warp owns
                        // 64 samples, two per lane, and a phi tile; 3: the warps share 64
                        // samples, two per lane, and split the blocks, a phi tile each
};

constexpr int kBatchWarps = 4;

// Per request: x and grad_phi transposed to [feature][Mpad] (row F of both is
// zero for padding elements and neutral nodes; columns >= M are zero), so a warp reads one
// feature of its 32 samples as one coalesced 128-byte line.
struct ReqDev {
    const float* XT;
    const float* GT;    // nullptr: forward only
    double* phi;
    int64_t M;
    int64_t Mpad;
    int32_t F;
    int32_t cat;        // categorical elements: always the NaN-aware variant
    const int* has_nan;
    int* status;
};

constexpr int kInlineSegs = 40;

struct BatchArgs {
    const SegDev* segs;   // nullptr: seg and req below (a call of one request)
    const ReqDev* reqs;
    int n_segs;
    int sub;              // blocks per staged sub-chunk
    int stage;            // records per staging buffer
    int pad;
    int64_t n_items;
    unsigned long long* counter;
    int64_t tile_floats;  // floats of the phi region (max over the launch's requests)
    QuadF q;
    SegDev seg[kInlineSegs];
    ReqDev req;
};

// samples per item for each mode
__host__ __device__ __forceinline__ int item_samples(int mode) {
    return mode == 3 ? 64 : mode == 2 ? 64 * kBatchWarps : 32;
}

// floats of the phi region a request needs in a mode
inline int64_t tile_floats_for(int mode, int F) {
    return mode >= 2 ? (int64_t)kBatchWarps * (F + 1) * kTileLd2 : (int64_t)(F + 1) * kTileLd;
}

inline size_t batch_smem_bytes(int64_t tile_floats, int stage) {
    const size_t off = ((size_t)tile_floats * 4 + 15) & ~(size_t)15;
    return off + 2 * (size_t)stage * sizeof(Rec32) + 16;
}

// Register classes.  A block's fused pass holds about 12 registers per shared
// element, 10 / 36 / 88 for a subtree of height 1 / 2 / 3 and 35 more: class 8 takes
// the small blocks (4 thread blocks of 128 threads per SM; those near 128
// registers run 2.7% faster in class 12, adjoint of 200 trees of depth 8), 12 what fits
// 168 (3), 16 the other exact widths (255, 2); the padded widths 20..32 are class
// 32 and each of 40, 48, 56 and 64 (which spill) is a class of its own.
__host__ __device__ constexpr int batch_class(int D, int h) {
    if (D > 32) return D;
    if (D > 16) return 32;
    const int regs = 12 * D + (h == 0 ? 0 : h == 1 ? 10 : h == 2 ? 36 : 88) + 35;
    return regs <= 90 ? 8 : regs <= 168 ? 12 : 16;
}
constexpr int batch_blocks(int cls) { return cls == 8 ? 4 : cls == 12 ? 3 : cls == 16 ? 2 : 1; }

template <int C, bool SP>
cudaError_t launch_batch_class(const BatchArgs& a, size_t smem, cudaStream_t st);

#if QTS_DEVICE_PARTS

struct ItemCtx {
    const SegDev& sg;
    const ReqDev& rq;
    int64_t p0, p1, s0;
    float* ps;
    Rec32 *st0, *st1;
    uint64_t* bars;
    uint32_t* s_phase;
    int* s_flag;
    int sub;
    const QuadF& q;
};

// phi of `n` samples from tiles of [feature][ld], `tiles` of them, into the output
__device__ __forceinline__ void flush_phi(const ReqDev& rq, const float* t, int tiles, int tile_elems, int ld,
                                          int64_t s0, int n, int first, int step) {
    for (int s = first; s < n && s0 + s < rq.M; s += step)
        for (int f = threadIdx.x & 31; f < rq.F; f += 32) {
            float v = 0.f;
            for (int w = 0; w < tiles; ++w) v += t[w * tile_elems + f * ld + s];
            if (v != 0.f) atomicAdd(&rq.phi[(s0 + s) * (rq.F + 1) + f], (double)v);
        }
}

template <int D, int H, bool SP>
__device__ __forceinline__ bool batch_item(const ItemCtx& c) {
    const SegDev& sg = c.sg;
    const ReqDev& rq = c.rq;
    const int F = rq.F;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool has_nan = *rq.has_nan != 0 || rq.cat != 0;
    constexpr int kSlots = D + blk_slots(H);
    constexpr int ld = SP ? kTileLd2 : kTileLd;
    const bool own = SP && sg.mode == 2;  // every warp has its own samples
    const int tile_elems = (F + 1) * ld;
    float* my = SP ? c.ps + warp * tile_elems : c.ps;
    const int64_t sw = own ? c.s0 + 64 * warp : c.s0;
    for (int idx = threadIdx.x; idx < (SP ? kBatchWarps : 1) * tile_elems; idx += blockDim.x) c.ps[idx] = 0.f;
    __syncthreads();
    bool ok;
    auto run = [&](auto&& body) {
        return stream_records<Rec32>(sg.rec, blk_stride(D, H), c.p0, c.p1, c.sub, c.st0, c.st1, c.bars, c.s_phase,
                                     c.s_flag, rq.status, body, own);
    };
    if constexpr (SP) {
        const BwdCols<true> xr{rq.XT, rq.Mpad, sw + 2 * lane}, gr{rq.GT, rq.Mpad, sw + 2 * lane};
        ok = run([&](int64_t p, const Rec32* r) {
            double* g = sg.g + p * kSlots;
            if (has_nan) bwd_block<D, H, true, true, kPhiPrivate>(r, xr, gr, my, lane, c.q, g);
            else bwd_block<D, H, false, true, kPhiPrivate>(r, xr, gr, my, lane, c.q, g);
        });
    } else if (rq.GT) {
        const BwdCols<false> xr{rq.XT, rq.Mpad, sw + lane}, gr{rq.GT, rq.Mpad, sw + lane};
        ok = run([&](int64_t p, const Rec32* r) {
            bwd_block<D, H, true, false, kPhiAtomic>(r, xr, gr, my, lane, c.q, sg.g + p * kSlots);
        });
    } else {
        const GlobalCols xr{rq.XT, rq.Mpad, sw + lane};
        ok = run([&](int64_t, const Rec32* r) { fwd_block<D, H, 4, true, kPhiAtomic>(r, xr, my, lane, c.q); });
    }
    if (!ok) return false;
    // stream_records ended on a block barrier: every warp's adds are in the tiles
    if (rq.phi) {
        if (own) flush_phi(rq, my, 1, tile_elems, ld, sw, 64, 0, 1);
        else flush_phi(rq, c.ps, SP ? kBatchWarps : 1, tile_elems, ld, c.s0, SP ? 64 : 32, warp, kBatchWarps);
    }
    __syncthreads();  // the tiles are rewritten by the next item
    return true;
}

// the (width, height) pairs of a class, as keys 4 D + h
template <int CLS, bool SP, int KEY>
__device__ __forceinline__ bool batch_dispatch(const ItemCtx& c) {
    constexpr int D = KEY / 4, H = KEY % 4;
    constexpr bool width = CLS <= 16 ? D <= 16 : CLS == 32 ? (D > 16 && D <= 32 && D % 4 == 0) : D == CLS;
    if constexpr (width && H <= blk_max_h(D) && batch_class(D, H) == CLS) {
        if (c.sg.D == D && c.sg.h == H) return batch_item<D, H, SP>(c);
    }
    if constexpr (KEY + 1 < 4 * (CLS <= 16 ? 17 : CLS == 32 ? 33 : CLS + 1)) return batch_dispatch<CLS, SP, KEY + 1>(c);
    else return false;
}

template <int CLS, bool SP>
__global__ void __launch_bounds__(128, batch_blocks(CLS)) batch_kernel(const __grid_constant__ BatchArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    float* ps = (float*)smem;
    const size_t off = ((size_t)a.tile_floats * 4 + 15) & ~(size_t)15;
    Rec32* st0 = (Rec32*)(smem + off);
    Rec32* st1 = st0 + a.stage;
    uint64_t* bars = (uint64_t*)(st1 + a.stage);
    __shared__ int s_flag;
    __shared__ uint32_t s_phase[2];
    __shared__ long long s_item;
    const SegDev* segs = a.segs ? a.segs : a.seg;
    if (threadIdx.x == 0) {
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        mbar_fence_init();
        s_phase[0] = s_phase[1] = 0;
    }
    __syncthreads();
    for (;;) {
        if (threadIdx.x == 0) s_item = (long long)atomicAdd(a.counter, 1ull);
        __syncthreads();
        const int64_t item = s_item;
        __syncthreads();
        if (item >= a.n_items) break;
        int lo = 0, hi = a.n_segs - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (segs[mid].item_begin <= item) lo = mid;
            else hi = mid - 1;
        }
        const SegDev sg = segs[lo];
        const ReqDev rq = a.segs ? a.reqs[sg.req] : a.req;
        const int64_t local = item - sg.item_begin;
        const int64_t p0 = (local / sg.n_tiles) * sg.per_item;
        const ItemCtx c{sg, rq, p0, imin64(p0 + sg.per_item, sg.n), (local % sg.n_tiles) * item_samples(sg.mode),
                        ps, st0, st1, bars, s_phase, &s_flag, a.sub, a.q};
        if (!batch_dispatch<CLS, SP, (CLS <= 16 ? 0 : CLS == 32 ? 80 : 4 * CLS)>(c))
            break;  // a bounded wait ran out: status is set, stop this thread block
    }
}

template <int C, bool SP>
cudaError_t launch_batch_class(const BatchArgs& a, size_t smem, cudaStream_t st) {
    auto k = batch_kernel<C, SP>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, 128, smem);
    if (e != cudaSuccess) return e;
    const int64_t blocks = std::min<int64_t>((int64_t)std::max(1, per_sm) * num_sms(), std::max<int64_t>(1, a.n_items));
    k<<<(unsigned)blocks, 128, smem, st>>>(a);
    return cudaGetLastError();
}

#define QTS_INST(C, SP) template cudaError_t launch_batch_class<C, SP>(const BatchArgs&, size_t, cudaStream_t);
#if QTS_IN_PART(1)
QTS_INST(8, true)
#endif
#if QTS_IN_PART(2)
QTS_INST(12, true)
#endif
#if QTS_IN_PART(3)
QTS_INST(16, true)
#endif
#if QTS_IN_PART(4)
QTS_INST(8, false)
#endif
#if QTS_IN_PART(5)
QTS_INST(12, false)
#endif
#if QTS_IN_PART(6)
QTS_INST(16, false)
#endif
#if QTS_IN_PART(7)
QTS_INST(32, false)
#endif
#if QTS_IN_PART(8)
QTS_INST(40, false)
#endif
#if QTS_IN_PART(9)
QTS_INST(48, false)
#endif
#if QTS_IN_PART(10)
QTS_INST(56, false)
#endif
#if QTS_IN_PART(11)
QTS_INST(64, false)
#endif
#undef QTS_INST

#endif  // QTS_DEVICE_PARTS

#if !QTS_HOST_PART
}  // namespace qts
#endif

#if QTS_HOST_PART

// Everything a call does around its persistent kernels, for all requests at
// once: each thread block finds its request and its part of that request's work by
// its index (a call of sixteen small requests spent two thirds of its time in
// about a hundred launches of 3 us each).
struct ReqWork {
    const float* X;
    const float* G;       // nullptr: forward only
    float *XT, *GT;       // transposed copies
    double* phi;          // or nullptr
    double *gb, *g;       // G = sum of grad_phi's last column (zero before the call's first
                          // kernel); adjoint sums
    int* flag;            // some x is NaN or +inf
    const BlockEntry* ent;
    const double *bias_leaf, *bias_z;
    double *d_leaf, *d_z;
    double bias;
    int64_t M, Mpad, n_g, n_ent, n_nodes;
    int64_t begin, bias_begin, ent_begin;  // first thread block in the three kernels
    int32_t F;
    int32_t pad;
};
constexpr int kInitChunk = 8192;    // doubles per thread block set to zero or E[f]
// samples per thread block of the sum G: one thread block for all of them was 3.2 of the
// 4.2 ms of an adjoint of one tree of depth 2 on 4,000,000 samples
constexpr int kSumChunk = 8192;
constexpr int kNodeChunk = 4096;    // nodes per thread block of batch_bias_kernel
constexpr int kEntryChunk = 4096;   // entries per thread block of batch_entries_kernel

inline int64_t chunks_of(int64_t n, int64_t c) { return (n + c - 1) / c; }
// thread blocks of batch_prepare_kernel for one request: transposed copies of X and
// G, phi, adjoint sums, G's last column
__host__ __device__ inline int64_t prepare_tiles(const ReqWork& w) { return w.Mpad / 32 * ((w.F + 32) / 32); }
inline int64_t prepare_blocks(const ReqWork& w) {
    return prepare_tiles(w) * (w.G ? 2 : 1) + (w.phi ? chunks_of(w.M * (w.F + 1), kInitChunk) : 0) +
           (w.G ? chunks_of(w.n_g, kInitChunk) + chunks_of(w.M, kSumChunk) : 0);
}

// out[c * Mpad + s] = in[s * ld + c] for c < ncols, s < M; zero elsewhere (up to
// row nrows - 1, column Mpad - 1).
__device__ __forceinline__ void transpose_tile(const float* __restrict__ in, int64_t M, int ncols, int64_t ld,
                                               float* __restrict__ out, int nrows, int64_t Mpad, int* has_nan,
                                               int64_t s0, int c0) {
    __shared__ float tile[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    int nan_seen = 0;
    for (int r = ty; r < 32; r += 8) {
        const int64_t s = s0 + r;
        const int c = c0 + tx;
        float v = 0.f;
        if (s < M && c < ncols) v = in[s * ld + c];
        nan_seen |= !(v < INFINITY);
        tile[r][tx] = v;
    }
    __syncthreads();
    for (int r = ty; r < 32; r += 8) {
        const int c = c0 + r;
        const int64_t s = s0 + tx;
        if (c < nrows && s < Mpad) out[(int64_t)c * Mpad + s] = tile[tx][r];
    }
    if (has_nan && nan_seen) atomicOr(has_nan, 1);
}

template <int64_t ReqWork::*BEGIN>
__device__ __forceinline__ const ReqWork& find_work(const ReqWork* w, int n) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (w[mid].*BEGIN <= (int64_t)blockIdx.x) lo = mid;
        else hi = mid - 1;
    }
    return w[lo];
}

struct WorkArgs {
    const ReqWork* many;  // nullptr: one
    int n;
    ReqWork one;
};

__global__ void __launch_bounds__(256) batch_prepare_kernel(const __grid_constant__ WorkArgs a) {
    const ReqWork& w = a.many ? find_work<&ReqWork::begin>(a.many, a.n) : a.one;
    int64_t k = (int64_t)blockIdx.x - w.begin;
    const int64_t tiles = prepare_tiles(w);
    const int rows = (w.F + 32) / 32;
    if (k < tiles) {
        transpose_tile(w.X, w.M, w.F, w.F, w.XT, w.F + 1, w.Mpad, w.flag, k / rows * 32, (int)(k % rows) * 32);
        return;
    }
    k -= tiles;
    if (w.G) {
        if (k < tiles) {
            // Row F stays zero: neutral nodes and padding name feature F, and the
            // weight of E[f] (column F of grad_phi) is no gradient of theirs.  In a
            // neutral node it cancels only to FP32 rounding between a leaf's two sums.
            transpose_tile(w.G, w.M, w.F, w.F + 1, w.GT, w.F + 1, w.Mpad, nullptr, k / rows * 32,
                           (int)(k % rows) * 32);
            return;
        }
        k -= tiles;
    }
    if (w.phi) {
        const int64_t n = w.M * (w.F + 1), c = (n + kInitChunk - 1) / kInitChunk;
        if (k < c) {
            const int64_t end = imin64(n, (k + 1) * kInitChunk);
            for (int64_t i = k * kInitChunk + threadIdx.x; i < end; i += blockDim.x)
                w.phi[i] = (i % (w.F + 1) == w.F) ? w.bias : 0.0;
            return;
        }
        k -= c;
    }
    const int64_t c = (w.n_g + kInitChunk - 1) / kInitChunk;
    if (k < c) {
        const int64_t end = imin64(w.n_g, (k + 1) * kInitChunk);
        for (int64_t i = k * kInitChunk + threadIdx.x; i < end; i += blockDim.x) w.g[i] = 0.0;
        return;
    }
    k -= c;
    double acc = 0.0;
    const int64_t end = imin64(w.M, (k + 1) * kSumChunk);
    for (int64_t s = k * kSumChunk + threadIdx.x; s < end; s += blockDim.x)
        acc += (double)w.G[s * (w.F + 1) + w.F];
    for (int off = 16; off >= 1; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    __shared__ double part[8];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int i = 0; i < 8; ++i) t += part[i];
        atomicAdd(w.gb, t);
    }
}

// Both gradients start at their share of E[f]'s, G times a constant per node, ...
__global__ void __launch_bounds__(256) batch_bias_kernel(const __grid_constant__ WorkArgs a) {
    const ReqWork& w = a.many ? find_work<&ReqWork::bias_begin>(a.many, a.n) : a.one;
    const int64_t k = (int64_t)blockIdx.x - w.bias_begin;
    const double G = *w.gb;
    const int64_t end = imin64(w.n_nodes, (k + 1) * kNodeChunk);
    for (int64_t i = k * kNodeChunk + threadIdx.x; i < end; i += blockDim.x) {
        w.d_leaf[i] = G * w.bias_leaf[i];
        w.d_z[i] = G * w.bias_z[i];
    }
}

// ... then every block's sums are chained to its leaves and edges.
__global__ void __launch_bounds__(256) batch_entries_kernel(const __grid_constant__ WorkArgs a) {
    const ReqWork& w = a.many ? find_work<&ReqWork::ent_begin>(a.many, a.n) : a.one;
    const int64_t k = (int64_t)blockIdx.x - w.ent_begin;
    const int64_t end = imin64(w.n_ent, (k + 1) * kEntryChunk);
    for (int64_t i = k * kEntryChunk + threadIdx.x; i < end; i += blockDim.x) {
        const BlockEntry e = w.ent[i];
        atomicAdd(((e.target & 1u) ? w.d_leaf : w.d_z) + (e.target >> 1), e.coef * w.g[e.slot]);
    }
}

// ------------------------------------------------------------- host side --

struct BatchPlan {
    std::vector<uint64_t> key;
    cudaGraphExec_t exec = nullptr;
    cudaGraph_t graph = nullptr;
    void* dev = nullptr;  // segments, requests, counters
    int kernels = 0;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;  // around the persistent kernel(s)
};

static std::mutex g_plan_mu;
static std::vector<BatchPlan*> g_plans;  // most recent last
static thread_local BatchPlan* g_last_plan = nullptr;
// cached graphs (a caller that launches each of many requests on its own keeps
// one plan per request)
constexpr size_t kMaxPlans = 256;

static void destroy_plan(BatchPlan* p) {
    if (p->ev0) cudaEventDestroy(p->ev0);
    if (p->ev1) cudaEventDestroy(p->ev1);
    if (p->exec) cudaGraphExecDestroy(p->exec);
    if (p->graph) cudaGraphDestroy(p->graph);
    if (p->dev) cudaFree(p->dev);
    delete p;
}

// drop every cached plan that mentions this ensemble (called before it is freed
// or its device memory moves)
void batch_forget(const qts_ensemble* e) {
    std::lock_guard<std::mutex> lk(g_plan_mu);
    const uint64_t id = (uint64_t)(uintptr_t)e;
    for (size_t i = 0; i < g_plans.size();) {
        const auto& k = g_plans[i]->key;
        if (std::find(k.begin(), k.end(), id) != k.end()) {
            cudaDeviceSynchronize();
            if (g_last_plan == g_plans[i]) g_last_plan = nullptr;
            destroy_plan(g_plans[i]);
            g_plans.erase(g_plans.begin() + i);
        } else {
            ++i;
        }
    }
}

// Workspace of one request in its ensemble: [adjoint sums (grad only)][XT][GT (grad only)][flag]
constexpr int kGradHead = 256;  // doubles before the adjoint sums
struct BatchWork {
    size_t grad_bytes, xt_off, gt_off, flag_off, total;
    int64_t Mpad;
};

static size_t align256(size_t x) { return (x + 255) / 256 * 256; }

static BatchWork batch_work(const qts_ensemble* e, int64_t M, int F, bool grad) {
    BatchWork w;
    w.Mpad = (M + 64 * kBatchWarps - 1) / (64 * kBatchWarps) * (64 * kBatchWarps);
    // G = sum of grad_phi's last column, the work counter, then the blocks' adjoint sums
    w.grad_bytes = grad ? align256(sizeof(double) * (size_t)(kGradHead + e->n_blk_slots)) : 0;
    const size_t tbytes = align256(sizeof(float) * (size_t)(F + 1) * (size_t)w.Mpad);
    w.xt_off = w.grad_bytes;
    w.gt_off = w.xt_off + tbytes;
    w.flag_off = w.gt_off + (grad ? tbytes : 0);
    w.total = w.flag_off + 256;
    return w;
}

static ReqWork request_work(const qts_request& R, char* base) {
    qts_ensemble* e = R.ens;
    const BatchWork bw = batch_work(e, R.M, R.F, R.grad_phi != nullptr);
    ReqWork w;
    std::memset(&w, 0, sizeof(w));
    w.X = R.X;
    w.G = R.grad_phi;
    w.XT = (float*)(base + bw.xt_off);
    w.GT = (float*)(base + bw.gt_off);
    w.phi = R.phi;
    w.flag = (int*)(base + bw.flag_off);
    w.bias = e->prep.bias;
    w.M = R.M;
    w.Mpad = bw.Mpad;
    w.F = R.F;
    if (R.grad_phi) {
        w.gb = (double*)base;
        w.g = (double*)base + kGradHead;
        w.n_g = e->n_blk_slots;
        w.ent = e->blkdev.ent;
        w.n_ent = e->blkdev.n_ent;
        w.bias_leaf = e->blkdev.bias_leaf;
        w.bias_z = e->blkdev.bias_z;
        w.n_nodes = e->n_nodes;
        w.d_leaf = R.d_leaf;
        w.d_z = R.d_z;
    }
    return w;
}

struct WorkBlocks {
    int64_t prepare = 0, bias = 0, entries = 0;
};

static void number_work(ReqWork& w, WorkBlocks* n) {
    w.begin = n->prepare;
    w.bias_begin = n->bias;
    w.ent_begin = n->entries;
    n->prepare += prepare_blocks(w);
    n->bias += chunks_of(w.n_nodes, kNodeChunk);
    n->entries += chunks_of(w.n_ent, kEntryChunk);
}

static ReqDev request_dev(const ReqWork& w, const qts_ensemble* e) {
    return {w.XT, w.G ? w.GT : nullptr, w.phi, w.M, w.Mpad, w.F, e->prep.has_cat ? 1 : 0, w.flag, e->d_status};
}

// Per-width launch choices that override the ensembles' own while tuning: blocks per
// work item (0: the default rule), packed sample mapping (0: keep), and optionally
// only the buckets of one width.
struct BatchOverride {
    int paths[kMaxD + 1];
    int mode[kMaxD + 1];
    int only_width;
};

struct SegHost {
    SegDev d;
    double unit;   // cost of one block (all samples of one item)
    int cls;
    int64_t tile;  // floats of its phi region
    int bin;       // tile-size bin: one launch per (class, bin, rule)
    int nq;        // quadrature points of the bucket (QTS_NQ_EXACT: ceil(width / 2))
    int npad;      // ... padded to `pad`, what its variant of the pass takes per register pass
    int pad;
    int stride;
};

constexpr int kBatchSub = 16;  // blocks per staged sub-chunk

// Blocks per item of the default launch, from the work of the whole launch: two
// dozen items per resident thread block evens out the tail and serves small
// requests; at least 32 blocks keep the tile set-up and the phi flush (about
// 64 F atomics) small beside the sweeps, and 2,048 are plenty.
static void default_items(std::vector<SegHost>& segs) {
    double total = 0.0;
    for (const SegHost& s : segs) total += s.unit * (double)s.d.n * s.d.n_tiles;
    const double share = total / (24.0 * 2.5 * num_sms());
    for (SegHost& s : segs) {
        if (s.d.per_item > 0) continue;
        const double per = std::min(2048.0, std::max(32.0, share / s.unit));
        s.d.per_item = (int32_t)(((int64_t)per + 15) / 16 * 16);
    }
}

// The segments of one request's buckets; base: its workspace.
static void request_segments(const qts_request& R, char* base, int req, int n_quad, const BatchOverride* ov,
                             std::vector<SegHost>* out) {
    qts_ensemble* e = R.ens;
    const bool grad = R.grad_phi != nullptr;
    double* g = grad ? (double*)base + kGradHead : nullptr;
    for (const BlockBucket& b : e->blk) {
        const Tune& tn = e->tune[b.D];
        SegHost s;
        s.cls = batch_class(b.D, b.h);
        s.stride = blk_stride(b.D, b.h);
        int mode = 0;
        if (grad && b.D <= 16 && batch_smem_bytes(tile_floats_for(2, R.F), kBatchSub * s.stride) <= kSmemMax / 2) {
            // the warps share 64 samples and split the blocks; the tuner may
            // prefer 64 samples per warp on large requests
            const int want = ov && ov->mode[b.D] ? ov->mode[b.D] : tn.bt_mode;
            mode = want == 2 ? 2 : 3;
        }
        const int per = item_samples(mode);
        s.d.rec = e->blkdev.rec + b.rec_off;
        s.d.g = grad ? g + b.slot_off : nullptr;
        s.d.n = b.n;
        s.d.item_begin = 0;
        s.d.D = b.D;
        s.d.h = b.h;
        s.d.per_item = ov ? ov->paths[b.D] : tn.bt_paths;
        s.d.n_tiles = (int)((R.M + per - 1) / per);
        s.d.req = req;
        s.d.mode = mode;
        s.nq = nodes_for(n_quad, b.dmax, 1);
        // the pass of two samples per lane takes one node at a time, the others pairs,
        // the forward alone four
        const int pad = mode >= 2 ? 1 : grad ? 2 : 4;
        s.pad = pad;
        s.npad = (s.nq + pad - 1) / pad * pad;
        s.unit = blk_cost(b.D, b.h) * (grad ? 2.5 : 1.0) * s.npad / 8.0 * (mode == 0 ? 1.0 : per / 32.0);
        // a launch sizes its shared memory for its widest tile, and whatever
        // shared memory a thread block does not take stays L1 (which serves the x and
        // grad_phi loads): requests of one class are launched by tile size
        s.tile = tile_floats_for(mode, R.F);
        const int64_t tb = s.tile * 4;
        s.bin = tb <= 48 * 1024 ? 0 : tb <= 80 * 1024 ? 1 : 2;
        out->push_back(s);
    }
}

// A forward-only request that fills the chip by itself: the forward's own kernels, with
// phi tiles of the warps' own and a variant without NaN tests, in place of items.  8 trees of
// depth 18, F = 24, 2,000 samples: 6,934 us as items, 3,021 here (5,782 on the path
// tables); four of 100 trees of depth 8, F = 30, 2,000 samples 1,606 -> 755.  Below about 25 us
// of work its launches would weigh: small requests share the persistent kernels.
static bool forward_alone(const qts_request& R) {
    if (R.grad_phi || R.M <= 0) return false;
    double work = 0.0;
    for (const BlockBucket& b : R.ens->blk) work += (double)b.n * blk_cost(b.D, b.h);
    return work * (double)((R.M + 31) / 32) >= 2e7;
}

struct LaunchHost {
    int cls, nq, npad, pad;
    bool sp;
    size_t first, count;  // segments
    int64_t items, tile;
    int stride;
};

// Order the segments - one launch per (class, tile bin, rule), heaviest items
// first within it - and number their items.
static std::vector<LaunchHost> order_segments(std::vector<SegHost>& segs, size_t max_segs) {
    default_items(segs);
    std::stable_sort(segs.begin(), segs.end(), [](const SegHost& a, const SegHost& b) {
        if (a.cls != b.cls) return a.cls > b.cls;
        if (a.pad != b.pad) return a.pad < b.pad;
        if (a.bin != b.bin) return a.bin < b.bin;
        if (a.npad != b.npad) return a.npad > b.npad;
        if (a.nq != b.nq) return a.nq > b.nq;
        return a.unit * a.d.per_item > b.unit * b.d.per_item;
    });
    std::vector<LaunchHost> out;
    for (size_t i = 0; i < segs.size(); ++i) {
        SegHost& s = segs[i];
        if (out.empty() || out.back().cls != s.cls || segs[i - 1].bin != s.bin || out.back().nq != s.nq ||
            out.back().npad != s.npad || out.back().pad != s.pad || out.back().count == max_segs)
            out.push_back({s.cls, s.nq, s.npad, s.pad, s.d.mode >= 2, i, 0, 0, 0, 0});
        LaunchHost& l = out.back();
        s.d.item_begin = l.items;
        l.items += (s.d.n + s.d.per_item - 1) / s.d.per_item * s.d.n_tiles;
        l.tile = std::max(l.tile, s.tile);
        l.stride = std::max(l.stride, s.stride);
        ++l.count;
    }
    return out;
}

// Launch one entry of order_segments; a.segs / a.seg and a.reqs / a.req are set.
static cudaError_t launch_ordered(const LaunchHost& l, BatchArgs& a, unsigned long long* counter, cudaStream_t st) {
    a.n_segs = (int)l.count;
    a.n_items = l.items;
    a.counter = counter;
    a.tile_floats = std::max<int64_t>(l.tile, kTileLd);
    a.sub = kBatchSub;
    // wide inputs: stage fewer blocks at a time until the thread block fits
    while (a.sub > 1 && batch_smem_bytes(a.tile_floats, a.sub * l.stride) > kSmemMax) a.sub /= 2;
    a.stage = a.sub * l.stride;
    a.pad = 0;
    if (!make_quad(l.nq, &a.q, nullptr, l.pad) || a.q.n_pad != l.npad) return cudaErrorInvalidValue;
    const size_t smem = batch_smem_bytes(a.tile_floats, a.stage);
    if (smem > kSmemMax) return cudaErrorInvalidConfiguration;
    if (l.sp) {
        switch (l.cls) {
            case 8: return launch_batch_class<8, true>(a, smem, st);
            case 12: return launch_batch_class<12, true>(a, smem, st);
            case 16: return launch_batch_class<16, true>(a, smem, st);
            default: return cudaErrorInvalidValue;
        }
    }
    switch (l.cls) {
        case 8: return launch_batch_class<8, false>(a, smem, st);
        case 12: return launch_batch_class<12, false>(a, smem, st);
        case 16: return launch_batch_class<16, false>(a, smem, st);
        case 32: return launch_batch_class<32, false>(a, smem, st);
        case 40: return launch_batch_class<40, false>(a, smem, st);
        case 48: return launch_batch_class<48, false>(a, smem, st);
        case 56: return launch_batch_class<56, false>(a, smem, st);
        default: return launch_batch_class<64, false>(a, smem, st);
    }
}

constexpr size_t kBatchBranches = 8;  // parallel branches of persistent kernels in a graph

static qts_status build_plan(int n, const qts_request* reqs, int n_quad, BatchPlan* plan,
                             cudaStream_t cap, const BatchOverride* ov = nullptr) {
    std::vector<SegHost> segs;
    std::vector<ReqDev> rd(n);
    std::vector<ReqWork> rw(n);
    std::vector<int> alone;  // requests that run the forward's own kernels
    WorkBlocks nb;
    const size_t flag_bytes = 256 * ((sizeof(int) * (size_t)n + 255) / 256);
    const size_t gb_bytes = 256 * ((sizeof(double) * (size_t)n + 255) / 256);
    for (int r = 0; r < n; ++r) {
        const qts_request& R = reqs[r];
        char* ws = (char*)R.ens->d_work;
        rw[r] = request_work(R, ws);
        if (forward_alone(R)) {
            rw[r].Mpad = 0;  // no transposed copy
            if (!ov) alone.push_back(r);
        } else if (R.M > 0) {
            request_segments(R, ws, r, n_quad, ov, &segs);
        }
        number_work(rw[r], &nb);
    }
    default_items(segs);  // from the whole launch, also where one width of it is timed
    if (ov && ov->only_width > 0)
        segs.erase(std::remove_if(segs.begin(), segs.end(), [&](const SegHost& s) { return s.d.D != ov->only_width; }),
                   segs.end());
    const std::vector<LaunchHost> launches = order_segments(segs, (size_t)1 << 30);
    auto pad = [](size_t v) { return (v + 255) / 256 * 256; };
    const size_t seg_bytes = pad(sizeof(SegDev) * std::max<size_t>(segs.size(), 1));
    const size_t req_bytes = pad(sizeof(ReqDev) * (size_t)n), work_bytes = pad(sizeof(ReqWork) * (size_t)n);
    const size_t cnt_bytes = pad(sizeof(unsigned long long) * std::max<size_t>(launches.size(), 1));
    cudaError_t ce = cudaMalloc(&plan->dev, seg_bytes + req_bytes + work_bytes + cnt_bytes + flag_bytes + gb_bytes);
    if (ce != cudaSuccess) return cuda_fail(ce, "batch plan allocation");
    char* base = (char*)plan->dev;
    SegDev* d_segs = (SegDev*)base;
    ReqDev* d_reqs = (ReqDev*)(base + seg_bytes);
    ReqWork* d_work = (ReqWork*)(base + seg_bytes + req_bytes);
    unsigned long long* d_cnt = (unsigned long long*)(base + seg_bytes + req_bytes + work_bytes);
    int* d_flag = (int*)(base + seg_bytes + req_bytes + work_bytes + cnt_bytes);
    double* d_gb = (double*)((char*)d_flag + flag_bytes);
    for (int r = 0; r < n; ++r) {
        rw[r].flag = d_flag + r;
        rw[r].gb = d_gb + r;
        rd[r] = request_dev(rw[r], reqs[r].ens);
    }
    std::vector<SegDev> sd(segs.size());
    for (size_t i = 0; i < segs.size(); ++i) sd[i] = segs[i].d;
    if (!sd.empty()) ce = cudaMemcpy(d_segs, sd.data(), sizeof(SegDev) * sd.size(), cudaMemcpyHostToDevice);
    if (ce == cudaSuccess) ce = cudaMemcpy(d_reqs, rd.data(), sizeof(ReqDev) * n, cudaMemcpyHostToDevice);
    if (ce == cudaSuccess) ce = cudaMemcpy(d_work, rw.data(), sizeof(ReqWork) * n, cudaMemcpyHostToDevice);
    if (ce != cudaSuccess) return cuda_fail(ce, "batch plan upload");

    ce = cudaEventCreate(&plan->ev0);
    if (ce == cudaSuccess) ce = cudaEventCreate(&plan->ev1);
    if (ce != cudaSuccess) return cuda_fail(ce, "batch plan events");
    // capture: preparation, persistent kernels, epilogue.  The persistent kernels
    // (and the gradients' start values) are branches of the graph, so one class's
    // last items run beside the next one's first.
    std::vector<cudaStream_t> side(std::min<size_t>(launches.size() + alone.size(), kBatchBranches), nullptr);
    std::vector<cudaEvent_t> done(side.size() + 1, nullptr);
    for (auto& x : side)
        if (ce == cudaSuccess) ce = cudaStreamCreateWithFlags(&x, cudaStreamNonBlocking);
    for (auto& x : done)
        if (ce == cudaSuccess) ce = cudaEventCreateWithFlags(&x, cudaEventDisableTiming);
    auto drop = [&] {
        for (auto& x : side)
            if (x) cudaStreamDestroy(x);
        for (auto& x : done)
            if (x) cudaEventDestroy(x);
    };
    if (ce == cudaSuccess) ce = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (ce != cudaSuccess) {
        drop();
        return cuda_fail(ce, "graph capture begin");
    }
    int kernels = 0;
    cudaError_t err = cudaSuccess;
    WorkArgs wa;
    std::memset(&wa, 0, sizeof(wa));
    wa.many = d_work;
    wa.n = n;
    auto work = [&](auto kernel, int64_t blocks, cudaStream_t st) {
        if (blocks <= 0 || err != cudaSuccess) return;
        if (blocks > 0x7fffffffLL) {
            err = cudaErrorInvalidConfiguration;
            return;
        }
        kernel<<<(unsigned)blocks, 256, 0, st>>>(wa);
        err = cudaGetLastError();
        ++kernels;
    };
    err = cudaMemsetAsync(d_cnt, 0, cnt_bytes + flag_bytes + gb_bytes, cap);
    work(batch_prepare_kernel, nb.prepare, cap);
    if (err == cudaSuccess) err = cudaEventRecordWithFlags(plan->ev0, cap, cudaEventRecordExternal);
    if (err == cudaSuccess) err = cudaEventRecord(done.back(), cap);
    for (size_t b = 0; b < side.size() && err == cudaSuccess; ++b) err = cudaStreamWaitEvent(side[b], done.back(), 0);
    for (size_t c = 0; c < launches.size() && err == cudaSuccess; ++c) {
        BatchArgs a;
        a.segs = d_segs + launches[c].first;
        a.reqs = d_reqs;
        err = launch_ordered(launches[c], a, d_cnt + c, side[c % side.size()]);
        ++kernels;
    }
    for (size_t i = 0; i < alone.size() && err == cudaSuccess; ++i) {
        const qts_request& R = reqs[alone[i]];
        err = launch_fwd_blocks(R.ens, R.X, R.M, R.F, n_quad, R.phi, side[(launches.size() + i) % side.size()], &kernels);
    }
    work(batch_bias_kernel, nb.bias, cap);
    for (size_t b = 0; b < side.size(); ++b) {
        // join every branch, also after an error: the capture must end whole
        cudaError_t j = cudaEventRecord(done[b], side[b]);
        if (j == cudaSuccess) j = cudaStreamWaitEvent(cap, done[b], 0);
        if (err == cudaSuccess) err = j;
    }
    if (err == cudaSuccess) err = cudaEventRecordWithFlags(plan->ev1, cap, cudaEventRecordExternal);
    work(batch_entries_kernel, nb.entries, cap);
    cudaGraph_t g = nullptr;
    ce = cudaStreamEndCapture(cap, &g);
    drop();
    if (err != cudaSuccess) {
        if (g) cudaGraphDestroy(g);
        return cuda_fail(err, "batched launch during capture");
    }
    if (ce != cudaSuccess) return cuda_fail(ce, "graph capture end");
    plan->graph = g;
    ce = cudaGraphInstantiate(&plan->exec, g, 0);
    if (ce != cudaSuccess) return cuda_fail(ce, "graph instantiate");
    plan->kernels = kernels;
    return QTS_OK;
}

static thread_local int g_last_batch_kernels = 0;

}  // namespace qts

using namespace qts;

namespace qts {

// Argument checks shared by the batched call and its tuner; grows every
// request's workspace to what the batched launch needs.
static qts_status check_batch(int32_t n, const qts_request* reqs, int32_t n_quad) {
    if (n < 1 || !reqs) return fail(QTS_ERR_ARG, "no requests");
    for (int r = 0; r < n; ++r) {
        const qts_request& R = reqs[r];
        qts_status st = check_call(R.ens, R.X, R.M, R.F, n_quad);
        if (st != QTS_OK) return fail(st, "request " + std::to_string(r) + ": " + qts_last_error());
        if (R.ens->flags & QTS_FLAG_FP64)
            return fail(QTS_ERR_UNSUPPORTED, "request " + std::to_string(r) + ": batched calls use FP32 tables");
        if (!R.grad_phi && !R.phi) return fail(QTS_ERR_ARG, "request " + std::to_string(r) + ": nothing to compute");
        if (R.grad_phi && (!R.d_leaf || !R.d_z))
            return fail(QTS_ERR_ARG, "request " + std::to_string(r) + ": d_leaf/d_z are NULL");
        for (int s = 0; s < r; ++s)
            if (reqs[s].ens == R.ens)
                return fail(QTS_ERR_ARG, "an ensemble may appear in at most one request of a batch");
    }
    for (int r = 0; r < n; ++r) {
        const qts_request& R = reqs[r];
        qts_status st = ensure_blocks(R.ens, R.grad_phi != nullptr);
        if (st != QTS_OK) return st;
        // (a graph launch cannot be captured, so the workspace stays the library's)
        st = ensure_workspace_uncaptured(R.ens, batch_work(R.ens, R.M, R.F, R.grad_phi != nullptr).total);
        if (st != QTS_OK) return st;
    }
    return QTS_OK;
}

}  // namespace qts

extern "C" qts_status qts_batched_fwd_bwd(int32_t n, const qts_request* reqs, int32_t n_quad,
                                          qts_stream_t stream) try {
    {
        const qts_status st = check_batch(n, reqs, n_quad);
        if (st != QTS_OK) return st;
    }
    std::vector<uint64_t> key;
    key.push_back((uint64_t)n_quad);
    for (int r = 0; r < n; ++r) {
        const qts_request& R = reqs[r];
        for (uint64_t v : {(uint64_t)(uintptr_t)R.ens, (uint64_t)(uintptr_t)R.X, (uint64_t)R.M, (uint64_t)R.F,
                           (uint64_t)(uintptr_t)R.grad_phi, (uint64_t)(uintptr_t)R.phi,
                           (uint64_t)(uintptr_t)R.d_leaf, (uint64_t)(uintptr_t)R.d_z,
                           (uint64_t)(uintptr_t)R.ens->d_work, (uint64_t)(uintptr_t)R.ens->blkdev.rec,
                           (uint64_t)R.ens->tune_gen})
            key.push_back(v);
    }
    cudaGraphExec_t exec = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_plan_mu);
        for (size_t i = 0; i < g_plans.size(); ++i) {
            if (g_plans[i]->key == key) {
                BatchPlan* p = g_plans[i];
                g_plans.erase(g_plans.begin() + i);
                g_plans.push_back(p);
                exec = p->exec;
                g_last_batch_kernels = p->kernels;
                g_last_plan = p;
                break;
            }
        }
    }
    if (!exec) {
        cudaStream_t cap;
        cudaError_t ce = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
        if (ce != cudaSuccess) return cuda_fail(ce, "capture stream");
        auto* plan = new BatchPlan();
        plan->key = key;
        qts_status st = build_plan(n, reqs, n_quad, plan, cap);
        cudaStreamDestroy(cap);
        if (st != QTS_OK) {
            destroy_plan(plan);
            return st;
        }
        std::lock_guard<std::mutex> lk(g_plan_mu);
        if (g_plans.size() >= kMaxPlans) {
            cudaDeviceSynchronize();
            if (g_last_plan == g_plans.front()) g_last_plan = nullptr;
            destroy_plan(g_plans.front());
            g_plans.erase(g_plans.begin());
        }
        g_plans.push_back(plan);
        exec = plan->exec;
        g_last_batch_kernels = plan->kernels;
        g_last_plan = plan;
    }
    cudaError_t ce = cudaGraphLaunch(exec, (cudaStream_t)stream);
    if (ce != cudaSuccess) return cuda_fail(ce, "graph launch");
    return QTS_OK;
} QTS_ENTRY_END

namespace qts {

// Device time of the persistent kernels of one plan built for `reqs` with the
// override `ov` (the faster of two launches after a first); the plan is destroyed
// afterwards.
static qts_status time_plan(int n, const qts_request* reqs, int n_quad, const BatchOverride& ov,
                            cudaStream_t cap, cudaStream_t st, float* ms) {
    auto* plan = new BatchPlan();
    qts_status s = build_plan(n, reqs, n_quad, plan, cap, &ov);
    cudaError_t ce = cudaSuccess;
    *ms = 1e30f;
    for (int k = 0; k < 3 && s == QTS_OK && ce == cudaSuccess; ++k) {
        float t = 0.f;
        ce = cudaGraphLaunch(plan->exec, st);
        if (ce == cudaSuccess) ce = cudaEventSynchronize(plan->ev1);
        if (ce == cudaSuccess) ce = cudaEventElapsedTime(&t, plan->ev0, plan->ev1);
        if (k > 0) *ms = std::min(*ms, t);
    }
    if (s == QTS_OK && ce != cudaSuccess) s = cuda_fail(ce, "batched tuning run");
    cudaStreamSynchronize(st);
    destroy_plan(plan);
    return s;
}

}  // namespace qts

extern "C" qts_status qts_batched_autotune(int32_t n, const qts_request* reqs, int32_t n_quad, int64_t max_samples,
                                           int32_t* chosen, qts_stream_t stream) try {
    qts_status st = check_batch(n, reqs, n_quad);
    if (st != QTS_OK) return st;
    if (max_samples < 0) return fail(QTS_ERR_ARG, "max_samples must be >= 0");
    std::vector<qts_request> sub(reqs, reqs + n);
    if (max_samples > 0)
        for (auto& R : sub) R.M = std::min<int64_t>(R.M, max_samples);
    // work per bucket width of the reduced batch, and whether the width runs the
    // pass of two samples per lane for some request
    std::vector<double> work(kMaxD + 1, 0.0);
    std::vector<char> packed(kMaxD + 1, 0);
    for (const auto& R : sub) {
        if (R.M <= 0 || forward_alone(R)) continue;
        for (const BlockBucket& b : R.ens->blk) {
            work[b.D] += (double)R.M * (double)b.n * blk_cost(b.D, b.h);
            if (R.grad_phi && b.D <= 16) packed[b.D] = 1;
        }
    }
    double total = 0.0;
    for (double w : work) total += w;
    std::vector<int> widths;
    for (int D = 1; D <= kMaxD; ++D)
        if (work[D] > 0.01 * total) widths.push_back(D);  // the rest keep the defaults
    std::sort(widths.begin(), widths.end(), [&](int a, int b) { return work[a] > work[b]; });
    cudaStream_t cap;
    cudaError_t ce = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
    if (ce != cudaSuccess) return cuda_fail(ce, "capture stream");
    std::vector<int> best_paths(kMaxD + 1, 0), best_mode(kMaxD + 1, 0);
    for (int D : widths) {
        BatchOverride ov;
        std::memset(&ov, 0, sizeof(ov));
        ov.only_width = D;
        // the defaults first: they stay unless another choice is faster
        float best = 1e30f;
        for (int mode : {3, 2}) {
            if (mode == 2 && !packed[D]) continue;
            for (int paths : {0, 64, 256, 1024, 2048}) {
                ov.paths[D] = paths;
                ov.mode[D] = packed[D] ? mode : 0;
                float ms = 0.f;
                st = time_plan(n, sub.data(), n_quad, ov, cap, (cudaStream_t)stream, &ms);
                if (st != QTS_OK) {
                    cudaStreamDestroy(cap);
                    return st;
                }
                if (ms < best) {
                    best = ms;
                    best_paths[D] = paths;
                    best_mode[D] = ov.mode[D];
                }
            }
        }
    }
    cudaStreamDestroy(cap);
    for (int r = 0; r < n; ++r) {
        qts_ensemble* e = reqs[r].ens;
        for (int D : widths) {
            e->tune[D].bt_paths = best_paths[D];
            e->tune[D].bt_mode = best_mode[D];
        }
        ++e->tune_gen;
        batch_forget(e);
    }
    if (chosen) {
        // widths that keep the default rule report what it gives for these requests
        std::vector<SegHost> segs;
        BatchOverride rule;
        std::memset(&rule, 0, sizeof(rule));
        for (const auto& R : sub)
            if (R.M > 0 && !forward_alone(R)) request_segments(R, (char*)R.ens->d_work, 0, n_quad, &rule, &segs);
        default_items(segs);
        for (int D : widths)
            for (const SegHost& s : segs)
                if (best_paths[D] == 0 && s.d.D == D) best_paths[D] = s.d.per_item;
        for (int D = 0; D <= kMaxD; ++D) {
            chosen[3 * D] = best_paths[D];
            chosen[3 * D + 1] = best_mode[D];
            chosen[3 * D + 2] = 0;
        }
    }
    return QTS_OK;
} QTS_ENTRY_END

extern "C" qts_status qts_get_batch_info(qts_ensemble* e, int64_t* n_paths, int64_t* sum_unique,
                                         int64_t* n_pair_paths, int32_t* n_buckets, int32_t* bucket_width,
                                         int64_t* bucket_paths) try {
    if (!e) return fail(QTS_ERR_ARG, "ensemble handle is NULL");
    if (e->flags & QTS_FLAG_FP64) return fail(QTS_ERR_UNSUPPORTED, "batched calls use FP32 tables");
    const qts_status st = ensure_pairs(e, false);
    if (st != QTS_OK) return st;
    if (n_paths) *n_paths = e->pair_sizes.n_paths;
    if (sum_unique) *sum_unique = e->pair_sizes.sum_unique;
    if (n_pair_paths) *n_pair_paths = e->pair_sizes.n_pair_paths;
    const size_t nb = std::min<size_t>(e->pair_sizes.buckets.size(), 32);
    if (n_buckets) *n_buckets = (int32_t)nb;
    for (size_t i = 0; i < nb; ++i) {
        if (bucket_width) bucket_width[i] = e->pair_sizes.buckets[i].D;
        if (bucket_paths) bucket_paths[i] = e->pair_sizes.buckets[i].n_paths;
    }
    return QTS_OK;
} QTS_ENTRY_END

// Adjoint of one request by the batched kernels, without a graph (qts_shap_backward).
// The samples go through in slabs, one after the other, so that their transposed
// copies stay small beside X and grad_phi, whatever M is.  A slab of 256 MiB (658,000
// samples at F = 50, 40,000 at F = 832) is many times what fills the chip.
namespace qts {

constexpr size_t kSlabBytes = (size_t)256 << 20;

int64_t adjoint_slab(int64_t M, int F) {
    constexpr int64_t unit = 64 * kBatchWarps;
    const int64_t s = (int64_t)(kSlabBytes / (2 * sizeof(float) * (size_t)(F + 1))) / unit * unit;
    return std::min(M, std::max(s, unit));
}

int64_t smaller_slab(int64_t slab) {
    constexpr int64_t unit = 64 * kBatchWarps;
    return slab <= unit ? 0 : std::max(unit, slab / 4 / unit * unit);
}

size_t adjoint_work_bytes(const qts_ensemble* e, int64_t slab, int F) { return batch_work(e, slab, F, true).total; }

cudaError_t launch_adjoint_blocks(qts_ensemble* e, void* work, int64_t slab, const float* X, const float* grad,
                                  int64_t M, int F, int n_quad, double* d_leaf, double* d_z, cudaStream_t st) {
    qts_request R;
    std::memset(&R, 0, sizeof(R));
    R.ens = e;
    R.F = F;
    R.d_leaf = d_leaf;
    R.d_z = d_z;
    cudaError_t err = cudaSuccess;
    WorkArgs wa;
    wa.many = nullptr;
    wa.n = 1;
    for (int64_t s0 = 0; s0 < M && err == cudaSuccess; s0 += slab) {
        R.X = X + s0 * F;
        R.grad_phi = grad + s0 * (F + 1);
        R.M = std::min(slab, M - s0);
        wa.one = request_work(R, (char*)work);
        if (s0 > 0) wa.one.n_g = 0;  // the sums go on from the slab before
        WorkBlocks nb;
        number_work(wa.one, &nb);
        if (nb.prepare > 0x7fffffffLL || nb.bias > 0x7fffffffLL || nb.entries > 0x7fffffffLL)
            return cudaErrorInvalidConfiguration;
        std::vector<SegHost> segs;
        request_segments(R, (char*)work, 0, n_quad, nullptr, &segs);
        const std::vector<LaunchHost> launches = order_segments(segs, kInlineSegs);
        if (launches.size() > kGradHead - 1) return cudaErrorInvalidConfiguration;
        // the head before the sums: G (of all slabs), then a counter per launch
        unsigned long long* counter = (unsigned long long*)wa.one.gb + 1;
        if (s0 == 0) err = cudaMemsetAsync(wa.one.gb, 0, kGradHead * sizeof(double), st);
        else err = cudaMemsetAsync(counter, 0, (kGradHead - 1) * sizeof(double), st);
        if (err == cudaSuccess) err = cudaMemsetAsync(wa.one.flag, 0, sizeof(int), st);
        if (err != cudaSuccess) return err;
        batch_prepare_kernel<<<(unsigned)nb.prepare, 256, 0, st>>>(wa);
        err = cudaGetLastError();
        for (size_t c = 0; c < launches.size() && err == cudaSuccess; ++c) {
            BatchArgs a;
            a.segs = nullptr;
            a.reqs = nullptr;
            for (size_t i = 0; i < launches[c].count; ++i) a.seg[i] = segs[launches[c].first + i].d;
            a.req = request_dev(wa.one, e);
            err = launch_ordered(launches[c], a, counter + c, st);
        }
    }
    if (err == cudaSuccess) {
        batch_bias_kernel<<<(unsigned)chunks_of(wa.one.n_nodes, kNodeChunk), 256, 0, st>>>(wa);
        err = cudaGetLastError();
    }
    if (err == cudaSuccess && wa.one.n_ent > 0) {
        batch_entries_kernel<<<(unsigned)chunks_of(wa.one.n_ent, kEntryChunk), 256, 0, st>>>(wa);
        err = cudaGetLastError();
    }
    return err;
}

}  // namespace qts

extern "C" qts_status qts_get_block_info(qts_ensemble* e, int64_t* n_blocks, int64_t* elements, int64_t* inner_nodes,
                                         int64_t* pair_nodes) try {
    if (!e) return fail(QTS_ERR_ARG, "ensemble handle is NULL");
    const qts_status st = ensure_blocks(e, false);
    if (st != QTS_OK) return st;
    int64_t v[4] = {0, 0, 0, 0};
    for (const BlockBucket& b : e->blk) {
        v[0] += b.n;
        v[1] += b.n * b.D;
        v[2] += b.n * blk_inner(b.h);
        v[3] += b.n * blk_pairs(b.h);
    }
    if (n_blocks) *n_blocks = v[0];
    if (elements) *elements = v[1];
    if (inner_nodes) *inner_nodes = v[2];
    if (pair_nodes) *pair_nodes = v[3];
    return QTS_OK;
} QTS_ENTRY_END

extern "C" int32_t qts_batched_kernel_count(void) { return g_last_batch_kernels; }

extern "C" qts_status qts_batched_last_kernel_ms(float* ms) {
    if (!ms) return fail(QTS_ERR_ARG, "ms is NULL");
    std::lock_guard<std::mutex> lk(g_plan_mu);
    if (!g_last_plan || std::find(g_plans.begin(), g_plans.end(), g_last_plan) == g_plans.end())
        return fail(QTS_ERR_ARG, "no batched call on this thread");
    cudaError_t ce = cudaEventSynchronize(g_last_plan->ev1);
    if (ce == cudaSuccess) ce = cudaEventElapsedTime(ms, g_last_plan->ev0, g_last_plan->ev1);
    return ce == cudaSuccess ? QTS_OK : cuda_fail(ce, "batched kernel timing");
}

#endif  // QTS_HOST_PART
