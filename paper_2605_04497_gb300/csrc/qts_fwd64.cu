// First-order Shapley values in FP64 (QTS_FLAG_FP64) on the block tables.
//
// The layout of qts_fwd_blocks.cu (32 samples per thread block, the warps split its
// blocks), with the weights, leaf values and all products in FP64, one quadrature
// node at a time.  Bound by the FP64 pipe, which takes two fused multiply-adds per
// SM and clock: what counts is the number of FP64 operations, and the blocks need
// about a fifth of what one path per leaf does.  50 trees of depth 6 (3,094 leaves, F =
// 13), 700 samples: 2.29 ms on the path tables, 0.29 ms here.
//
// qts-build-parts: 6 (part 0: host code; parts 1-5: one register class each)
#include <algorithm>

#include "qts_blocks.cuh"

namespace qts {

constexpr int k64Segs = 40;
constexpr int k64Warps = 4;

struct Seg64 {
    const Rec32* rec;
    const double* dbl;
    int64_t n;
    int64_t cta_begin;  // first thread block
    int32_t per_cta;    // blocks per thread block
    int32_t D, h;
};

struct Args64 {
    Seg64 seg[k64Segs];
    QuadD q;
    int n_seg;
    int n_tiles;   // sample tiles of 32
    int F;
    int tile;      // phi tiles in shared memory, one per warp; 0: they would not fit,
                   // contributions go straight to phi with atomics
    const float* X;
    int64_t M;
    double* phi;
};

__host__ __device__ constexpr int c64_class(int D) { return D <= 6 ? 0 : D <= 10 ? 1 : D <= 16 ? 2 : D <= 32 ? 3 : 4; }
[[maybe_unused]] constexpr int k64Classes = 5;

template <int CLS>
cudaError_t launch_64(const Args64& a, int64_t ctas, size_t smem, cudaStream_t st);

#if QTS_DEVICE_PARTS

struct Phi64 {
    double* tile;  // this warp's phi tile, or nullptr
    double* row;   // this lane's row of the output (tile = nullptr)
    int F, lane;
    bool live;
    __device__ __forceinline__ void add(int f, double v) const {
        if (tile) tile[f * kTileLd + lane] += v;
        else if (live && f < F && v != 0.0) atomicAdd(&row[f], v);
    }
};

template <int H, int D>
struct Tree64 {
    const Rec32* nodes;
    const double* q;  // the block's FP64 values
    double d[2 * blk_inner(H) + blk_pairs(H) + 1];    // o - z of the inner nodes' edges; val d of the pairs
    double acc[blk_inner(H) + blk_pairs(H) + 1];      // sum over the quadrature nodes
    static constexpr int pair_at(int n) { return 2 * blk_inner(H) + n - 1 - blk_inner(H); }

    template <int N, int LEVELS>
    __device__ __forceinline__ void decode(const SmemCols& xr) {
        const float4 b = rec4(nodes + blk_rec(H, N) + 1);
        bool l, r;
        node_sides<N == 1, true>(xr(feat_of(__float_as_uint(b.w))), b, &l, &r);
        const double* z = q + blk_dbl(D, H, N);
        acc[N - 1] = 0.0;
        if constexpr (LEVELS == 1) {
            d[pair_at(N)] = z[0] * ((l ? 1.0 : 0.0) - z[2]) + z[1] * ((r ? 1.0 : 0.0) - z[3]);
        } else {
            d[2 * (N - 1)] = (l ? 1.0 : 0.0) - z[0];
            d[2 * (N - 1) + 1] = (r ? 1.0 : 0.0) - z[1];
            decode<2 * N, LEVELS - 1>(xr);
            decode<2 * N + 1, LEVELS - 1>(xr);
        }
    }
    template <int N, int LEVELS>
    __device__ __forceinline__ double eval(double t, double C) {
        const double* z = q + blk_dbl(D, H, N);
        if constexpr (LEVELS == 1) {
            acc[N - 1] += C;
            return fma(t, d[pair_at(N)], z[4]);
        } else {
            const double dl = d[2 * (N - 1)], dr = d[2 * (N - 1) + 1];
            const double al = fma(t, dl, z[0]), ar = fma(t, dr, z[1]);
            const double gl = eval<2 * N, LEVELS - 1>(t, C * al);
            const double gr = eval<2 * N + 1, LEVELS - 1>(t, C * ar);
            acc[N - 1] = fma(C, fma(dl, gl, dr * gr), acc[N - 1]);
            return fma(al, gl, ar * gr);
        }
    }
    template <int N, int LEVELS>
    __device__ __forceinline__ void finish(const Phi64& phi) const {
        const int f = feat_of(nodes[blk_rec(H, N) + 1].bits);
        if constexpr (LEVELS == 1) {
            phi.add(f, d[pair_at(N)] * acc[N - 1]);
        } else {
            phi.add(f, acc[N - 1]);
            finish<2 * N, LEVELS - 1>(phi);
            finish<2 * N + 1, LEVELS - 1>(phi);
        }
    }
};

template <int D, int H>
__device__ __forceinline__ void block64(const Rec32* __restrict__ r, const double* __restrict__ z, const SmemCols& xr,
                                        const Phi64& phi, const QuadD& q) {
    constexpr int DN = D > 0 ? D : 1;
    const uint32_t* words = reinterpret_cast<const uint32_t*>(r + 1 + D);
    double d[DN], acc[DN];
    Tree64<H, D> t;
    t.nodes = r + blk_head(D);
    t.q = z;
#pragma unroll
    for (int j = 0; j < D; ++j) {
        const float4 e = rec4(r + 1 + j);
        const uint32_t word = words[j];
        d[j] = (satisfies<true>(xr(feat_of(word)), e.z, e.w, word) ? 1.0 : 0.0) - z[1 + j];
        acc[j] = 0.0;
    }
    if constexpr (H > 0) t.template decode<1, H>(xr);
#pragma unroll 1
    for (int m = 0; m < q.n; ++m) {
        const double tm = q.t[m];
        double A[DN], P[D + 1], G;
        P[0] = q.w[m];
#pragma unroll
        for (int j = 0; j < D; ++j) {
            A[j] = fma(tm, d[j], z[1 + j]);
            P[j + 1] = P[j] * A[j];
        }
        if constexpr (H > 0) G = t.template eval<1, H>(tm, P[D]);
        else G = z[0];
#pragma unroll
        for (int j = D - 1; j >= 0; --j) {
            acc[j] = fma(P[j], G, acc[j]);
            if (j > 0) G *= A[j];
        }
    }
#pragma unroll
    for (int j = 0; j < D; ++j) phi.add(feat_of(words[j]), d[j] * acc[j]);
    if constexpr (H > 0) t.template finish<1, H>(phi);
}

template <int D, int H>
__device__ __forceinline__ void run64(const Args64& a, const Seg64& sg, int64_t p0, int64_t p1, const SmemCols& xr,
                                      const Phi64& phi) {
    for (int64_t p = p0 + (threadIdx.x >> 5); p < p1; p += k64Warps)
        block64<D, H>(sg.rec + p * blk_stride(D, H), sg.dbl + p * blk_doubles(D, H), xr, phi, a.q);
}

template <int D>
__device__ __forceinline__ void segment64(const Args64& a, const Seg64& sg, int64_t p0, int64_t p1,
                                          const SmemCols& xr, const Phi64& phi) {
    if constexpr (blk_max_h(D) >= 3) {
        if (sg.h == 3) return run64<D, 3>(a, sg, p0, p1, xr, phi);
    }
    if constexpr (blk_max_h(D) >= 2) {
        if (sg.h == 2) return run64<D, 2>(a, sg, p0, p1, xr, phi);
    }
    if (sg.h == 1) return run64<D, 1>(a, sg, p0, p1, xr, phi);
    run64<D, 0>(a, sg, p0, p1, xr, phi);
}

template <int CLS>
__global__ void __launch_bounds__(k64Warps * 32) fwd64_kernel(const __grid_constant__ Args64 a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int F = a.F;
    const int stride = (F + 1) * kTileLd;
    double* ps = (double*)smem;
    float* xs = (float*)(ps + (a.tile ? k64Warps * stride : 0));
    int si = 0;
    while (si + 1 < a.n_seg && (int64_t)blockIdx.x >= a.seg[si + 1].cta_begin) ++si;
    const Seg64 sg = a.seg[si];
    const int64_t local = (int64_t)blockIdx.x - sg.cta_begin;
    const int64_t s0 = (local % a.n_tiles) * 32;
    const int64_t p0 = (local / a.n_tiles) * sg.per_cta;
    const int64_t p1 = imin64(p0 + sg.per_cta, sg.n);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (a.tile)
        for (int idx = threadIdx.x; idx < k64Warps * stride; idx += blockDim.x) ps[idx] = 0.0;
    (void)load_tile_t(xs, a.X, s0, a.M, F, F, 1);
    const bool live = s0 + lane < a.M;
    const SmemCols xr{xs, lane};
    const Phi64 phi{a.tile ? ps + warp * stride : nullptr, a.phi + (live ? (s0 + lane) * (F + 1) : 0), F, lane, live};
#define QTS_CASE(DD) \
    case DD: segment64<DD>(a, sg, p0, p1, xr, phi); break;
    if constexpr (CLS == 0) {
        switch (sg.D) {
            QTS_CASE(0) QTS_CASE(1) QTS_CASE(2) QTS_CASE(3) QTS_CASE(4) QTS_CASE(5) QTS_CASE(6)
            default: break;
        }
    } else if constexpr (CLS == 1) {
        switch (sg.D) {
            QTS_CASE(7) QTS_CASE(8) QTS_CASE(9) QTS_CASE(10)
            default: break;
        }
    } else if constexpr (CLS == 2) {
        switch (sg.D) {
            QTS_CASE(11) QTS_CASE(12) QTS_CASE(13) QTS_CASE(14) QTS_CASE(15) QTS_CASE(16)
            default: break;
        }
    } else if constexpr (CLS == 3) {
        switch (sg.D) {
            QTS_CASE(20) QTS_CASE(24) QTS_CASE(28) QTS_CASE(32)
            default: break;
        }
    } else {
        switch (sg.D) {
            QTS_CASE(40) QTS_CASE(48) QTS_CASE(56) QTS_CASE(64)
            default: break;
        }
    }
#undef QTS_CASE
    if (!a.tile) return;
    __syncthreads();
    for (int s = warp; s < 32 && s0 + s < a.M; s += k64Warps)
        for (int f = lane; f < F; f += 32) {
            double v = 0.0;
            for (int w = 0; w < k64Warps; ++w) v += ps[w * stride + f * kTileLd + s];
            if (v != 0.0) atomicAdd(&a.phi[(s0 + s) * (F + 1) + f], v);
        }
}

template <int CLS>
cudaError_t launch_64(const Args64& a, int64_t ctas, size_t smem, cudaStream_t st) {
    auto k = fwd64_kernel<CLS>;
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    k<<<(unsigned)ctas, k64Warps * 32, smem, st>>>(a);
    return cudaGetLastError();
}

#define QTS_INST(C) template cudaError_t launch_64<C>(const Args64&, int64_t, size_t, cudaStream_t);
#if QTS_IN_PART(1)
QTS_INST(0)
#endif
#if QTS_IN_PART(2)
QTS_INST(1)
#endif
#if QTS_IN_PART(3)
QTS_INST(2)
#endif
#if QTS_IN_PART(4)
QTS_INST(3)
#endif
#if QTS_IN_PART(5)
QTS_INST(4)
#endif
#undef QTS_INST

#endif  // QTS_DEVICE_PARTS

#if !QTS_HOST_PART
}  // namespace qts
#endif

#if QTS_HOST_PART

cudaError_t launch_fwd64(const qts_ensemble* e, const float* X, int64_t M, int F, int n_quad, double* phi,
                         cudaStream_t st) {
    if (M <= 0) return cudaSuccess;
    const int64_t tiles = (M + 31) / 32;
    // phi tiles while a thread block leaves room for another on its SM
    const size_t rows = (size_t)(F + 1) * kTileLd;
    const bool tile = rows * (k64Warps * sizeof(double) + sizeof(float)) <= 110 * 1024;
    const size_t smem = rows * ((tile ? k64Warps * sizeof(double) : 0) + sizeof(float));
    double total = 0.0;
    for (const BlockBucket& b : e->blk) total += (double)b.n * blk_cost(b.D, b.h);
    total *= (double)tiles;
    for (int cls = 0; cls < k64Classes; ++cls) {
        for (int nq = n_quad == QTS_NQ_EXACT ? QTS_MAX_QUAD : n_quad; nq >= (n_quad == QTS_NQ_EXACT ? 1 : n_quad); --nq) {  // one launch per rule of the class
            Args64 a;
            a.n_seg = 0;
            a.n_tiles = (int)tiles;
            a.F = F;
            a.tile = tile ? 1 : 0;
            a.X = X;
            a.M = M;
            a.phi = phi;
            int64_t ctas = 0;
            auto flush = [&]() -> cudaError_t {
                if (a.n_seg == 0) return cudaSuccess;
                if (ctas > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
                const cudaError_t r = cls == 0   ? launch_64<0>(a, ctas, smem, st)
                                      : cls == 1 ? launch_64<1>(a, ctas, smem, st)
                                      : cls == 2 ? launch_64<2>(a, ctas, smem, st)
                                      : cls == 3 ? launch_64<3>(a, ctas, smem, st)
                                                 : launch_64<4>(a, ctas, smem, st);
                a.n_seg = 0;
                ctas = 0;
                return r;
            };
            // the FP64 pipe is busy with few warps: two dozen thread blocks per SM
            // even out the tail, and one round of the warps is the least
            const double share = std::min(400e3, total / (24.0 * num_sms()));
            bool made = false;
            for (auto it = e->blk.rbegin(); it != e->blk.rend(); ++it) {  // wide blocks first
                const BlockBucket& b = *it;
                if (c64_class(b.D) != cls || nodes_for(n_quad, b.dmax, 1) != nq) continue;
                if (!made && !make_quad(nq, nullptr, &a.q, 1)) return cudaErrorInvalidValue;
                made = true;
                if (a.n_seg == k64Segs) {
                    const cudaError_t r = flush();
                    if (r != cudaSuccess) return r;
                }
                const int64_t per = std::max<int64_t>(k64Warps, (int64_t)(share / blk_cost(b.D, b.h)));
                Seg64& sg = a.seg[a.n_seg++];
                sg = {e->blkdev.rec + b.rec_off, e->blkdev.dbl + b.dbl_off, b.n, ctas,
                      (int32_t)((per + k64Warps - 1) / k64Warps * k64Warps), b.D, b.h};
                ctas += (b.n + sg.per_cta - 1) / sg.per_cta * tiles;
            }
            const cudaError_t r = flush();
            if (r != cudaSuccess) return r;
        }
    }
    return cudaSuccess;
}

}  // namespace qts

#endif  // QTS_HOST_PART
