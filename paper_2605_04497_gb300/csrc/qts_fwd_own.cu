// First-order Shapley values of many samples under a small ensemble, FP32.
//
// The forward of qts_fwd_blocks.cu gives every (bucket, tile of 32 samples) a thread
// block of its own; when the ensemble has few blocks, setting it up (tiles, barrier,
// staging, flush) costs more than they do.  Here a thread block stages all blocks of a
// class of widths once and its warps, each with tiles of its own, walk them for one
// tile of 32 samples after another, without a barrier of the thread block.
//
// Bound by instruction issue, as there.  Thread block per (bucket, tile) before and
// here: one tree of depth 4, 200,000 samples, F = 12 213 -> 31 us (one launch per path
// width of the path tables: 66); five of depth 6, F = 40 929 -> 280 (508); one of depth
// 10, 20,000 samples, F = 12 195 -> 180 (182); five of depth 3, 1,000,000 samples, F = 2
// 864 -> 92 (164).
//
// qts-build-parts: 9 (part 0: host code; parts 1-8: the kernels)
#include <algorithm>

#include "qts_blocks.cuh"

namespace qts {

constexpr int kOwnWarps = 4;

struct OwnSeg {
    const Rec32* rec;
    int32_t n;
    int32_t D, h;
};

struct OwnArgs {
    OwnSeg seg[kFbSegs];
    QuadF q;
    int n_seg;
    int records;   // of all segments
    int F;
    int cat;       // ensemble has categorical elements: always the NaN-aware variant
    int64_t n_tiles;
    const float* X;
    int64_t M;
    double* phi;
    int* status;
};

template <int CLS, int NP>
cudaError_t launch_own(const OwnArgs& a, size_t smem, cudaStream_t st);

#if QTS_DEVICE_PARTS

template <int D, int H, int NP>
__device__ __forceinline__ void own_run(const OwnArgs& a, const Rec32* buf, int n, bool has_nan, const float* xs,
                                        float* ps) {
    const int lane = threadIdx.x & 31;
    const SmemCols xr{xs, lane};
    for (int i = 0; i < n; ++i) {
        const Rec32* r = buf + i * blk_stride(D, H);
        if (has_nan) fwd_block<D, H, NP, true, kPhiPrivate>(r, xr, ps, lane, a.q);
        else fwd_block<D, H, NP, false, kPhiPrivate>(r, xr, ps, lane, a.q);
    }
}

template <int D, int NP>
__device__ __forceinline__ void own_segment(const OwnArgs& a, int h, const Rec32* buf, int n, bool has_nan,
                                            const float* xs, float* ps) {
    if constexpr (blk_max_h(D) >= 3) {
        if (h == 3) return own_run<D, 3, NP>(a, buf, n, has_nan, xs, ps);
    }
    if constexpr (blk_max_h(D) >= 2) {
        if (h == 2) return own_run<D, 2, NP>(a, buf, n, has_nan, xs, ps);
    }
    if (h == 1) return own_run<D, 1, NP>(a, buf, n, has_nan, xs, ps);
    own_run<D, 0, NP>(a, buf, n, has_nan, xs, ps);
}

template <int CLS, int NP>
__global__ void __launch_bounds__(kOwnWarps * 32, CLS <= 3 ? 4 : 2) fwd_own_kernel(const __grid_constant__ OwnArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_flag;
    const int F = a.F;
    const int rows = (F + 1) * kTileLd;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float* xs = (float*)smem + 2 * warp * rows;
    float* ps = xs + rows;
    Rec32* recs = (Rec32*)(smem + (((size_t)2 * kOwnWarps * rows * 4 + 15) & ~(size_t)15));
    uint64_t* bar = (uint64_t*)(recs + a.records);
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        mbar_fence_init();
        mbar_arrive_expect_tx(bar, (uint32_t)a.records * (uint32_t)sizeof(Rec32));
        Rec32* to = recs;
        for (int k = 0; k < a.n_seg; ++k) {
            const int len = a.seg[k].n * blk_stride(a.seg[k].D, a.seg[k].h);
            bulk_g2s(to, a.seg[k].rec, (uint32_t)len * (uint32_t)sizeof(Rec32), bar);
            to += len;
        }
        s_flag = mbar_wait_bounded(bar, 0) ? 1 : 0;
        if (!s_flag) {
            report(a.status, QTS_ERR_TIMEOUT);
            (void)mbar_wait_bounded(bar, 0);  // its own copies, still in flight
        }
    }
    __syncthreads();
    if (!s_flag) return;
    (void)mbar_try_wait(bar, 0);  // acquire the bulk-copy writes
    for (int64_t t = (int64_t)blockIdx.x * kOwnWarps + warp; t < a.n_tiles; t += (int64_t)gridDim.x * kOwnWarps) {
        const int64_t s0 = t * 32;
        int nan_seen = 0;
        for (int idx = lane; idx < 32 * F; idx += 32) {
            const int s = idx / F, c = idx - s * F;
            const float v = s0 + s < a.M ? a.X[(s0 + s) * F + c] : 0.f;
            xs[c * kTileLd + s] = v;
            nan_seen |= !(v < INFINITY);
        }
        for (int idx = lane; idx < kTileLd; idx += 32) xs[F * kTileLd + idx] = 0.f;
        for (int idx = lane; idx < rows; idx += 32) ps[idx] = 0.f;
        const bool has_nan = __any_sync(0xffffffffu, nan_seen) || a.cat != 0;
        __syncwarp();
        const Rec32* buf = recs;
        for (int k = 0; k < a.n_seg; ++k) {
            const int D = a.seg[k].D, h = a.seg[k].h, n = a.seg[k].n;
#define QTS_CASE(DD) \
    case DD: own_segment<DD, NP>(a, h, buf, n, has_nan, xs, ps); break;
            if constexpr (CLS == 0) {
                switch (D) {
                    QTS_CASE(0) QTS_CASE(1) QTS_CASE(2) QTS_CASE(3) QTS_CASE(4) QTS_CASE(5)
                    default: break;
                }
            } else if constexpr (CLS == 1) {
                switch (D) {
                    QTS_CASE(6) QTS_CASE(7) QTS_CASE(8)
                    default: break;
                }
            } else if constexpr (CLS == 2) {
                switch (D) {
                    QTS_CASE(9) QTS_CASE(10) QTS_CASE(11) QTS_CASE(12)
                    default: break;
                }
            } else if constexpr (CLS == 3) {
                switch (D) {
                    QTS_CASE(13) QTS_CASE(14) QTS_CASE(15) QTS_CASE(16)
                    default: break;
                }
            } else {
                switch (D) {
                    QTS_CASE(20) QTS_CASE(24) QTS_CASE(28) QTS_CASE(32) QTS_CASE(40) QTS_CASE(48) QTS_CASE(56)
                    QTS_CASE(64)
                    default: break;
                }
            }
#undef QTS_CASE
            buf += n * blk_stride(D, h);
        }
        __syncwarp();
        for (int idx = lane; idx < 32 * F; idx += 32) {
            const int s = idx / F, f = idx - s * F;
            const float v = ps[f * kTileLd + s];
            if (s0 + s < a.M && v != 0.f) atomicAdd(&a.phi[(s0 + s) * (F + 1) + f], (double)v);
        }
        __syncwarp();  // the tiles are rewritten for the next 32 samples
    }
}

template <int CLS, int NP>
cudaError_t launch_own(const OwnArgs& a, size_t smem, cudaStream_t st) {
    auto k = fwd_own_kernel<CLS, NP>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kOwnWarps * 32, smem);
    if (e != cudaSuccess) return e;
    const int64_t blocks = std::min<int64_t>((int64_t)std::max(1, per_sm) * num_sms(),
                                             (a.n_tiles + kOwnWarps - 1) / kOwnWarps);
    k<<<(unsigned)blocks, kOwnWarps * 32, smem, st>>>(a);
    return cudaGetLastError();
}

#define QTS_INST(C, N) template cudaError_t launch_own<C, N>(const OwnArgs&, size_t, cudaStream_t);
#if QTS_IN_PART(1)
QTS_INST(0, 8)
#endif
#if QTS_IN_PART(2)
QTS_INST(0, 4)
#endif
#if QTS_IN_PART(3)
QTS_INST(0, 2)
#endif
#if QTS_IN_PART(4)
QTS_INST(1, 4)
#endif
#if QTS_IN_PART(5)
QTS_INST(1, 2)
#endif
#if QTS_IN_PART(6)
QTS_INST(2, 2)
#endif
#if QTS_IN_PART(7)
QTS_INST(3, 2)
#endif
#if QTS_IN_PART(8)
QTS_INST(4, 2)
#endif
#undef QTS_INST

#endif  // QTS_DEVICE_PARTS

#if !QTS_HOST_PART
}  // namespace qts
#endif

#if QTS_HOST_PART

static size_t own_smem(int F, int64_t records) {
    const size_t tiles = ((size_t)2 * kOwnWarps * (F + 1) * kTileLd * 4 + 15) & ~(size_t)15;
    return tiles + (size_t)records * sizeof(Rec32) + sizeof(uint64_t);
}

// Whether one launch over these buckets takes less time here than with a thread block
// per (bucket, tile).  Two thread blocks per SM have to fit; then by a model of both,
// in warp instructions (blk_cost): a warp alone on its scheduler issues one in about
// 1.4 ns, the chip 790 in 1 ns, and a thread block over there costs 6.7 ns of the chip.
// Measured with 0.5, 1, 1.4 and 2 ns on 1 to 10 trees of depth 2 to 13, 1,000 to 20,000
// samples: 0.5 takes calls here that lose up to 1.8 times (ten trees of depth 6,
// 8,000 samples, F = 3: 64 us against 35), 2 leaves gains of up to 1.37 times (two of depth
// 8, 20,000 samples, F = 40: 101 against 137); at 1.4 none of these calls is slower
// than over there by more than its noise.
bool fwd_own_wins(const BlockBucket* const* pick, int n_pick, int64_t M, int F) {
    int64_t records = 0;
    double cost = 0.0;
    for (int k = 0; k < n_pick; ++k) {
        if (pick[k]->n > 4096) return false;
        records += pick[k]->n * blk_stride(pick[k]->D, pick[k]->h);
        cost += (double)pick[k]->n * blk_cost(pick[k]->D, pick[k]->h);
    }
    if (own_smem(F, records) > 110 * 1024) return false;
    const double tiles = (double)((M + 31) / 32);
    return 2000.0 + 1.4 * cost <= tiles * (6.7 * n_pick + cost / 790.0);
}

cudaError_t launch_fwd_own(const qts_ensemble* e, const float* X, int64_t M, int F, int cls, int nq, int np,
                           const BlockBucket* const* pick, int n_pick, double* phi, cudaStream_t st) {
    OwnArgs a;
    if (n_pick > kFbSegs || !make_quad(nq, &a.q, nullptr, 2)) return cudaErrorInvalidValue;
    a.n_seg = 0;
    a.records = 0;
    for (int k = 0; k < n_pick; ++k) {
        const BlockBucket* b = pick[k];
        a.seg[a.n_seg++] = {e->blkdev.rec + b->rec_off, (int32_t)b->n, b->D, b->h};
        a.records += (int)b->n * blk_stride(b->D, b->h);
    }
    a.F = F;
    a.cat = e->prep.has_cat ? 1 : 0;
    a.n_tiles = (M + 31) / 32;
    a.X = X;
    a.M = M;
    a.phi = phi;
    a.status = e->d_status;
    const size_t smem = own_smem(F, a.records);
#define QTS_GO(C, N) \
    if (cls == C && np == N) return launch_own<C, N>(a, smem, st);
    QTS_GO(0, 8) QTS_GO(0, 4) QTS_GO(0, 2) QTS_GO(1, 4) QTS_GO(1, 2) QTS_GO(2, 2)
    QTS_GO(3, 2) QTS_GO(4, 2)
#undef QTS_GO
    return cudaErrorInvalidValue;
}

}  // namespace qts

#endif  // QTS_HOST_PART
