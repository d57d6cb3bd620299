// First-order Shapley values of a few samples (M <= kFewRows) on the block tables.
//
// With one sample per lane a call on one row would leave 31 of 32 lanes idle, so
// here lane l holds the pair (block l / M, sample l mod M): a warp takes 32 / M
// blocks of one bucket at a time, which all have the same shape, so its lanes
// stay together.  Each lane reads its own block's records from global memory
// (the loads of a block are independent of each other), and phi goes to one
// shared tile with atomics.  All buckets of a class of widths are one launch.
//
// Bound by latency: 300 trees of depth 8 (71,759 leaves, F = 50), one row: 113 us
// as one launch per path width on the path tables, 38 us with three classes of widths, 30 us
// here, about 25 of them on the device.
//
// qts-build-parts: 4 (part 0: host code; parts 1-3: one class of widths each)
#include <algorithm>

#include "qts_blocks.cuh"

namespace qts {

constexpr int kFewSegs = 40;
constexpr int kFewWarps = 4;
constexpr int kFewNp = 4;  // quadrature nodes per pass (rules are padded to it)

struct FewSeg {
    const Rec32* rec;
    int64_t n;
    int64_t cta_begin;  // first thread block
    int32_t per_cta;    // blocks per thread block
    int32_t D, h;
};

struct FewArgs {
    FewSeg seg[kFewSegs];
    QuadF q;
    int n_seg;
    int F;
    int M;
    int group;  // 32 / M
    const float* X;
    double* phi;
};

__host__ __device__ constexpr int few_class(int D) { return D <= 8 ? 0 : D <= 16 ? 1 : 2; }
[[maybe_unused]] constexpr int kFewClasses = 3;

template <int CLS>
cudaError_t launch_few(const FewArgs& a, int64_t ctas, size_t smem, cudaStream_t st);

#if QTS_DEVICE_PARTS

template <int D, int H>
__device__ __forceinline__ void few_run(const FewArgs& a, const FewSeg& sg, int64_t p0, int64_t p1, const float* xs,
                                        float* ps) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int slot = lane / a.M, col = lane - slot * a.M;
    const SmemCols xr{xs, col};
    for (int64_t i = p0 + (int64_t)warp * a.group; i < p1; i += (int64_t)kFewWarps * a.group) {
        const int64_t k = i + slot;
        if (slot < a.group && k < p1)
            fwd_block<D, H, kFewNp, true, kPhiAtomicNz>(sg.rec + k * blk_stride(D, H), xr, ps, col, a.q);
    }
}

template <int D>
__device__ __forceinline__ void few_segment(const FewArgs& a, const FewSeg& sg, int64_t p0, int64_t p1,
                                            const float* xs, float* ps) {
    if constexpr (blk_max_h(D) >= 3) {
        if (sg.h == 3) return few_run<D, 3>(a, sg, p0, p1, xs, ps);
    }
    if constexpr (blk_max_h(D) >= 2) {
        if (sg.h == 2) return few_run<D, 2>(a, sg, p0, p1, xs, ps);
    }
    if (sg.h == 1) return few_run<D, 1>(a, sg, p0, p1, xs, ps);
    few_run<D, 0>(a, sg, p0, p1, xs, ps);
}

template <int CLS>
__global__ void __launch_bounds__(kFewWarps * 32) few_kernel(const __grid_constant__ FewArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int F = a.F;
    const int stride = (F + 1) * kTileLd;
    float* xs = (float*)smem;
    float* ps = xs + stride;
    int si = 0;
    while (si + 1 < a.n_seg && (int64_t)blockIdx.x >= a.seg[si + 1].cta_begin) ++si;
    const FewSeg sg = a.seg[si];
    const int64_t p0 = ((int64_t)blockIdx.x - sg.cta_begin) * sg.per_cta;
    const int64_t p1 = imin64(p0 + sg.per_cta, sg.n);
    // columns of the a.M samples only; row F is the padding elements' zero row
    for (int idx = threadIdx.x; idx < a.M * (F + 1); idx += blockDim.x) {
        const int s = idx / (F + 1), f = idx - s * (F + 1);
        xs[f * kTileLd + s] = f < F ? a.X[(int64_t)s * F + f] : 0.f;
        ps[f * kTileLd + s] = 0.f;
    }
    __syncthreads();
#define QTS_CASE(DD) \
    case DD: few_segment<DD>(a, sg, p0, p1, xs, ps); break;
    if constexpr (CLS == 0) {
        switch (sg.D) {
            QTS_CASE(0) QTS_CASE(1) QTS_CASE(2) QTS_CASE(3) QTS_CASE(4) QTS_CASE(5) QTS_CASE(6) QTS_CASE(7) QTS_CASE(8)
            default: break;
        }
    } else if constexpr (CLS == 1) {
        switch (sg.D) {
            QTS_CASE(9) QTS_CASE(10) QTS_CASE(11) QTS_CASE(12) QTS_CASE(13) QTS_CASE(14) QTS_CASE(15) QTS_CASE(16)
            default: break;
        }
    } else {
        switch (sg.D) {
            QTS_CASE(20) QTS_CASE(24) QTS_CASE(28) QTS_CASE(32) QTS_CASE(40) QTS_CASE(48) QTS_CASE(56) QTS_CASE(64)
            default: break;
        }
    }
#undef QTS_CASE
    __syncthreads();
    for (int idx = threadIdx.x; idx < a.M * F; idx += blockDim.x) {
        const int s = idx / F, f = idx - s * F;
        const float v = ps[f * kTileLd + s];
        if (v != 0.f) atomicAdd(&a.phi[(int64_t)s * (F + 1) + f], (double)v);
    }
}

template <int CLS>
cudaError_t launch_few(const FewArgs& a, int64_t ctas, size_t smem, cudaStream_t st) {
    auto k = few_kernel<CLS>;
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    k<<<(unsigned)ctas, kFewWarps * 32, smem, st>>>(a);
    return cudaGetLastError();
}

#define QTS_INST(C) template cudaError_t launch_few<C>(const FewArgs&, int64_t, size_t, cudaStream_t);
#if QTS_IN_PART(1)
QTS_INST(0)
#endif
#if QTS_IN_PART(2)
QTS_INST(1)
#endif
#if QTS_IN_PART(3)
QTS_INST(2)
#endif
#undef QTS_INST

#endif  // QTS_DEVICE_PARTS

#if !QTS_HOST_PART
}  // namespace qts
#endif

#if QTS_HOST_PART

cudaError_t launch_fwd_few(const qts_ensemble* e, const float* X, int64_t M, int F, int n_quad, double* phi,
                           cudaStream_t st) {
    if (M <= 0) return cudaSuccess;
    const int group = (int)(32 / M);
    const size_t smem = 2 * (size_t)(F + 1) * kTileLd * 4;
    for (int cls = 0; cls < kFewClasses; ++cls) {
        for (int nq = n_quad == QTS_NQ_EXACT ? QTS_MAX_QUAD : n_quad; nq >= (n_quad == QTS_NQ_EXACT ? 1 : n_quad); --nq) {  // one launch per rule of the class
            FewArgs a;
            a.n_seg = 0;
            a.F = F;
            a.M = (int)M;
            a.group = group;
            a.X = X;
            a.phi = phi;
            int64_t ctas = 0;
            auto flush = [&]() -> cudaError_t {
                if (a.n_seg == 0) return cudaSuccess;
                if (ctas > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
                const cudaError_t r = cls == 0   ? launch_few<0>(a, ctas, smem, st)
                                      : cls == 1 ? launch_few<1>(a, ctas, smem, st)
                                                 : launch_few<2>(a, ctas, smem, st);
                a.n_seg = 0;
                ctas = 0;
                return r;
            };
            bool made = false;
            for (const BlockBucket& b : e->blk) {
                if (few_class(b.D) != cls || nodes_for(n_quad, b.dmax, 1) != nq) continue;
                if (!made && !make_quad(nq, &a.q, nullptr, kFewNp)) return cudaErrorInvalidValue;
                made = true;
                if (a.n_seg == kFewSegs) {
                    const cudaError_t r = flush();
                    if (r != cudaSuccess) return r;
                }
                // one round of the thread block's lanes, or, for large
                // ensembles, what makes about four thread blocks per SM
                const int64_t round = (int64_t)kFewWarps * group;
                const int64_t rounds =
                    std::min<int64_t>(kMostBlocks / round, std::max<int64_t>(1, b.n / (round * 4 * num_sms())));
                FewSeg& sg = a.seg[a.n_seg++];
                sg = {e->blkdev.rec + b.rec_off, b.n, ctas, (int32_t)(round * rounds), b.D,
                      b.h};
                ctas += (b.n + sg.per_cta - 1) / sg.per_cta;
            }
            const cudaError_t r = flush();
            if (r != cudaSuccess) return r;
        }
    }
    return cudaSuccess;
}

}  // namespace qts

#endif  // QTS_HOST_PART
