// First-order Shapley values on the block tables (qts_blocks.h), the FP32
// forward of more than a few samples.
//
// A thread block owns 32 samples (lane = sample) and a run of blocks of one
// bucket; its warps share the samples' tile, split the blocks and add into a phi
// tile each (plain read-add-write), summed and flushed into the FP64 output once
// with atomics.  Records are staged by double-buffered bulk copies.  All buckets
// of a register class and pass width are one launch: the segment table rides in
// the kernel's parameters and a thread block finds its segment by its index, so
// a small ensemble costs one or two launches instead of one per width.
//
// Bound by instruction issue and FP32: at 1,000 trees of depth 8 (239,216 leaves,
// 10,000 samples, F = 50) the path tables needed 14.98 ms at about 150 warp
// instructions per leaf and 32 samples; the blocks take 8.34 ms (8.85 before
// staging 16 and more at a time; then at most two levels of splits per block: 11.0,
// one: about 15).  Tried on the way and
// slower: two samples per lane with a loop over the nodes (18-31 ms: 8 warps per
// SM and a chain of dependent products), shape flags tested per node instead of
// complete subtrees (13.0 ms), four nodes per pass at widths up to 5 (9.3 ms).
//
// qts-build-parts: 9 (part 0: host code; parts 1-8: the kernels)
#include <algorithm>

#include "qts_blocks.cuh"

namespace qts {

constexpr int kFbWarps = 4;

struct FbSeg {
    const Rec32* rec;
    int64_t n;
    int64_t cta_begin;  // first thread block
    int32_t per_cta;    // blocks per thread block
    int32_t D, h;
};

struct FbArgs {
    FbSeg seg[kFbSegs];
    QuadF q;
    int n_seg;
    int n_tiles;   // sample tiles of 32
    int sub;       // blocks per staged sub-chunk
    int stage;     // records per staging buffer
    int nphi;      // phi tiles: one per warp, or 1 (shared-memory atomics)
    int F;
    int cat;       // ensemble has categorical elements: always the NaN-aware variant
    const float* X;
    int64_t M;
    double* phi;
    int* status;
};

// Register classes by width; each runs NP quadrature nodes per pass: eight while the
// prefix products fit 128 registers, then four, and two from width 9 (depth 20, 8
// trees, 5,000 samples: 18.3 ms with four nodes at 166-243 registers, 17.7 with two
// at 128 and 16.7 with longer staging, where four thread blocks per SM make up for the second decoding).
__host__ __device__ constexpr int fb_class(int D) { return D <= 5 ? 0 : D <= 8 ? 1 : D <= 12 ? 2 : D <= 16 ? 3 : 4; }
[[maybe_unused]] constexpr int kFbClasses = 5;
// nodes per pass of a class for a rule of n_pad points (padded to pairs)
static inline int fb_np(int cls, int n_pad) {
    int np = cls == 0 ? 8 : cls == 1 ? 4 : 2;
    while (np > 2 && n_pad % np != 0) np /= 2;
    return np;
}

template <int CLS, int NP>
cudaError_t launch_fb(const FbArgs& a, int64_t ctas, size_t smem, cudaStream_t st);

#if QTS_DEVICE_PARTS

template <int D, int H, int NP>
__device__ __forceinline__ bool fb_run(const FbArgs& a, const FbSeg& sg, int64_t p0, int64_t p1, bool has_nan,
                                       const float* xs, float* ps, Rec32* st0, Rec32* st1, uint64_t* bars,
                                       uint32_t* s_phase, int* s_flag) {
    const int lane = threadIdx.x & 31;
    const SmemCols xr{xs, lane};
    return stream_records<Rec32>(
        sg.rec, blk_stride(D, H), p0, p1, a.sub, st0, st1, bars, s_phase, s_flag, a.status,
        [&](int64_t, const Rec32* r) {
            if (a.nphi > 1) {
                if (has_nan) fwd_block<D, H, NP, true, kPhiPrivate>(r, xr, ps, lane, a.q);
                else fwd_block<D, H, NP, false, kPhiPrivate>(r, xr, ps, lane, a.q);
            } else {
                fwd_block<D, H, NP, true, kPhiAtomic>(r, xr, ps, lane, a.q);
            }
        });
}

template <int D, int NP>
__device__ __forceinline__ bool fb_segment(const FbArgs& a, const FbSeg& sg, int64_t p0, int64_t p1, bool has_nan,
                                           const float* xs, float* ps, Rec32* st0, Rec32* st1, uint64_t* bars,
                                           uint32_t* s_phase, int* s_flag) {
    if constexpr (blk_max_h(D) >= 3) {
        if (sg.h == 3) return fb_run<D, 3, NP>(a, sg, p0, p1, has_nan, xs, ps, st0, st1, bars, s_phase, s_flag);
    }
    if constexpr (blk_max_h(D) >= 2) {
        if (sg.h == 2) return fb_run<D, 2, NP>(a, sg, p0, p1, has_nan, xs, ps, st0, st1, bars, s_phase, s_flag);
    }
    if (sg.h == 1) return fb_run<D, 1, NP>(a, sg, p0, p1, has_nan, xs, ps, st0, st1, bars, s_phase, s_flag);
    return fb_run<D, 0, NP>(a, sg, p0, p1, has_nan, xs, ps, st0, st1, bars, s_phase, s_flag);
}

template <int CLS, int NP>
__global__ void __launch_bounds__(kFbWarps * 32, CLS <= 3 ? 4 : 2)
    fwd_blocks_kernel(const __grid_constant__ FbArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int F = a.F;
    const int stride = (F + 1) * kTileLd;
    float* xs = (float*)smem;
    float* ps = xs + stride;
    Rec32* st0 = (Rec32*)(smem + (((size_t)(1 + a.nphi) * stride * 4 + 15) & ~(size_t)15));
    Rec32* st1 = st0 + a.stage;
    uint64_t* bars = (uint64_t*)(st1 + a.stage);
    __shared__ int s_flag;
    __shared__ uint32_t s_phase[2];
    int si = 0;
    while (si + 1 < a.n_seg && (int64_t)blockIdx.x >= a.seg[si + 1].cta_begin) ++si;
    const FbSeg sg = a.seg[si];
    const int64_t local = (int64_t)blockIdx.x - sg.cta_begin;
    const int64_t s0 = (local % a.n_tiles) * 32;
    const int64_t p0 = (local / a.n_tiles) * sg.per_cta;
    const int64_t p1 = imin64(p0 + sg.per_cta, sg.n);
    const int warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        mbar_fence_init();
        s_phase[0] = s_phase[1] = 0;
    }
    for (int idx = threadIdx.x; idx < a.nphi * stride; idx += blockDim.x) ps[idx] = 0.f;
    const bool has_nan = load_tile_t(xs, a.X, s0, a.M, F, F, 1) || a.cat != 0;
    float* my = a.nphi > 1 ? ps + warp * stride : ps;
    bool ok = false;
#define QTS_CASE(DD) \
    case DD: ok = fb_segment<DD, NP>(a, sg, p0, p1, has_nan, xs, my, st0, st1, bars, s_phase, &s_flag); break;
    if constexpr (CLS == 0) {
        switch (sg.D) {
            QTS_CASE(0) QTS_CASE(1) QTS_CASE(2) QTS_CASE(3) QTS_CASE(4) QTS_CASE(5)
            default: break;
        }
    } else if constexpr (CLS == 1) {
        switch (sg.D) {
            QTS_CASE(6) QTS_CASE(7) QTS_CASE(8)
            default: break;
        }
    } else if constexpr (CLS == 2) {
        switch (sg.D) {
            QTS_CASE(9) QTS_CASE(10) QTS_CASE(11) QTS_CASE(12)
            default: break;
        }
    } else if constexpr (CLS == 3) {
        switch (sg.D) {
            QTS_CASE(13) QTS_CASE(14) QTS_CASE(15) QTS_CASE(16)
            default: break;
        }
    } else {
        switch (sg.D) {
            QTS_CASE(20) QTS_CASE(24) QTS_CASE(28) QTS_CASE(32) QTS_CASE(40) QTS_CASE(48) QTS_CASE(56) QTS_CASE(64)
            default: break;
        }
    }
#undef QTS_CASE
    if (!ok) return;
    // stream_records ended on a block barrier: every warp's adds are in its tile
    for (int s = warp; s < 32 && s0 + s < a.M; s += kFbWarps)
        for (int f = threadIdx.x & 31; f < F; f += 32) {
            float v = 0.f;
            for (int w = 0; w < a.nphi; ++w) v += ps[w * stride + f * kTileLd + s];
            if (v != 0.f) atomicAdd(&a.phi[(s0 + s) * (F + 1) + f], (double)v);
        }
}

template <int CLS, int NP>
cudaError_t launch_fb(const FbArgs& a, int64_t ctas, size_t smem, cudaStream_t st) {
    auto k = fwd_blocks_kernel<CLS, NP>;
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    k<<<(unsigned)ctas, kFbWarps * 32, smem, st>>>(a);
    return cudaGetLastError();
}

#define QTS_INST(C, N) template cudaError_t launch_fb<C, N>(const FbArgs&, int64_t, size_t, cudaStream_t);
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

static size_t fb_smem(int F, int nphi, int stage) {
    const size_t tiles = ((size_t)(1 + nphi) * (F + 1) * kTileLd * 4 + 15) & ~(size_t)15;
    return tiles + 2 * (size_t)stage * sizeof(Rec32) + 2 * sizeof(uint64_t);
}

// phi[:, :F] = 0, phi[:, F] = E[f]
__global__ void phi_init_kernel(double* phi, int64_t M, int F, double bias) {
    const int64_t n = M * (F + 1);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        phi[i] = (i % (F + 1) == F) ? bias : 0.0;
}

cudaError_t launch_phi_init(double* phi, int64_t M, int F, double bias, cudaStream_t st) {
    if (M <= 0) return cudaSuccess;
    const int64_t n = M * (F + 1);
    const int blocks = (int)std::min<int64_t>((n + 255) / 256, 4 * 152);
    phi_init_kernel<<<blocks, 256, 0, st>>>(phi, M, F, bias);
    return cudaGetLastError();
}

// Work per thread block (units of blk_cost) below which zeroing, loading and flushing the
// tiles, rows of 32 samples for each feature, weighs too much beside the blocks.  With the
// factor 200, 100 trees of depth 8 on 2,000 samples: F = 100 345 -> 305 us, 200 561 -> 433,
// 400 1,118 -> 694, 784 3,527 -> 1,531 (100: 345, 516, 804, 1,783; 400: 256, 444, 658,
// 1,423, but 33 samples of 20 trees of depth 14 180 -> 205).
static double fb_least(int F) { return 200.0 * (F + 40); }

cudaError_t launch_fwd_blocks(const qts_ensemble* e, const float* X, int64_t M, int F, int n_quad, double* phi,
                              cudaStream_t st, int* kernels) {
    if (M <= 0) return cudaSuccess;
    const int64_t tiles = (M + 31) / 32;
    double total = 0.0;
    for (const BlockBucket& b : e->blk) total += (double)b.n * blk_cost(b.D, b.h);
    total *= (double)tiles;
    for (int cls = 0; cls < kFbClasses; ++cls) {
        // one launch per rule of the class (QTS_NQ_EXACT takes one per bucket)
        for (int nq = n_quad == QTS_NQ_EXACT ? QTS_MAX_QUAD : n_quad; nq >= (n_quad == QTS_NQ_EXACT ? 1 : n_quad); --nq) {
            FbArgs a;
            a.n_seg = 0;
            int64_t ctas = 0;
            int stage = 0;
            const BlockBucket* pick[kFbSegs];
            int n_pick = 0;
            for (const BlockBucket& b : e->blk)
                if (fb_class(b.D) == cls && nodes_for(n_quad, b.dmax, 1) == nq) {
                    if (n_pick == kFbSegs) return cudaErrorInvalidValue;
                    pick[n_pick++] = &b;
                }
            if (n_pick == 0) continue;
            if (kernels) ++*kernels;
            if (!make_quad(nq, &a.q, nullptr, 2)) return cudaErrorInvalidValue;
            const int np = fb_np(cls, a.q.n_pad);
            if (fwd_own_wins(pick, n_pick, M, F)) {
                const cudaError_t r = launch_fwd_own(e, X, M, F, cls, nq, np, pick, n_pick, phi, st);
                if (r != cudaSuccess) return r;
                continue;
            }
            std::sort(pick, pick + n_pick,
                      [](const BlockBucket* x, const BlockBucket* y) { return blk_cost(x->D, x->h) > blk_cost(y->D, y->h); });
            int max_stride = 0;
            for (int k = 0; k < n_pick; ++k) max_stride = std::max(max_stride, blk_stride(pick[k]->D, pick[k]->h));
            // tiles of phi: one per warp while that leaves two thread blocks per SM,
            // then a shared one with atomics.  Blocks staged at a time: the most
            // that keeps four thread blocks per SM (a staged sub-chunk ends on a
            // barrier: 8 instead of 16 cost 5% on 1,000 trees of depth 8), and for
            // wide inputs what fits at all
            a.nphi = fb_smem(F, kFbWarps, 8 * max_stride) <= 110 * 1024 ? kFbWarps : 1;
            a.sub = 32;
            while (a.sub > 8 && fb_smem(F, a.nphi, a.sub * max_stride) > 56 * 1024) a.sub /= 2;
            while (a.sub > 1 && fb_smem(F, a.nphi, a.sub * max_stride) > kSmemMax) a.sub /= 2;
            stage = a.sub * max_stride;
            const size_t smem = fb_smem(F, a.nphi, stage);
            if (smem > kSmemMax) return cudaErrorInvalidConfiguration;
            a.stage = stage;
            a.n_tiles = (int)tiles;
            a.F = F;
            a.cat = e->prep.has_cat ? 1 : 0;
            a.X = X;
            a.M = M;
            a.phi = phi;
            a.status = e->d_status;
            // work per thread block: about eight rounds of the whole chip, and what
            // keeps the tiles' set-up and flush small beside it as far as that leaves
            // two rounds of the thread blocks that fit
            const int resident = std::min(cls <= 3 ? 4 : 2, std::max(1, (int)(kSmemMax / (smem + 1024))));
            const double two_rounds = total / (2.0 * num_sms() * resident);
            // a tuned share (of another call's samples, maybe) leaves two rounds too
            const double share = e->bpaths > 0 ? std::min(kBlkUnit * e->bpaths, std::max(4e3, two_rounds))
                                               : std::min(400e3, std::max({4e3, std::min(fb_least(F), two_rounds),
                                                                           total / (8.0 * num_sms() * 4)}));
            for (int k = 0; k < n_pick; ++k) {
                const BlockBucket* b = pick[k];
                FbSeg& sg = a.seg[a.n_seg++];
                sg.rec = e->blkdev.rec + b->rec_off;
                sg.n = b->n;
                sg.D = b->D;
                sg.h = b->h;
                sg.cta_begin = ctas;
                const int64_t per = std::min<int64_t>(
                    kMostBlocks, std::max<int64_t>(kFbWarps, (int64_t)(share / blk_cost(b->D, b->h))));
                sg.per_cta = (int32_t)((per + kFbWarps - 1) / kFbWarps * kFbWarps);
                ctas += (b->n + sg.per_cta - 1) / sg.per_cta * tiles;
            }
            if (ctas > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
            cudaError_t r = cudaErrorInvalidValue;
#define QTS_GO(C, N) \
    if (cls == C && np == N) r = launch_fb<C, N>(a, ctas, smem, st);
            QTS_GO(0, 8) QTS_GO(0, 4) QTS_GO(0, 2) QTS_GO(1, 4) QTS_GO(1, 2) QTS_GO(2, 2)
            QTS_GO(3, 2) QTS_GO(4, 2)
#undef QTS_GO
            if (r != cudaSuccess) return r;
        }
    }
    return cudaSuccess;
}

}  // namespace qts

#endif  // QTS_HOST_PART
