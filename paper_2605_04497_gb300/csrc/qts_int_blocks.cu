// Pairwise Shapley interaction values (Thm 1 with S = {i, j}) on the block tables
// (qts_blocks.h).
//
// For a block let C = w_m prod of the shared elements' factors, G the subtree's leaf
// sum, and for a node u of the subtree V_u = d_L G_L + d_R G_R (val d for a pair
// node) and U_u = V_u times the factors of the edges between the block's root and u,
// all at the quadrature nodes.  Then
//     two shared elements     SII_ij  += d_i d_j sum_m C / (a_i a_j) G,
//     shared element, node    SII_iu  += d_i sum_m C / a_i U_u,
//     node above a node       SII_vu  += sum_m C (edges to v) d_v (edges between) V_u,
//     first order             phi_u   += sum_m C U_u,
// with the quotients formed as products (running products between the elements
// against stored suffixes, no division).  Per leaf of a full h = 3 block that is a
// third of the pair sums, and of the work for each, that one path per leaf pair needs.
//
// Per thread block (32 samples x a run of blocks of one bucket) pair sums and
// first-order sums go to shared FP32 tiles (atomics: the warps share them) and are
// flushed into FP64 accumulators in the workspace laid out [pair][sample] and
// [feature][sample]; launch_int_finalize writes the (F+1) x (F+1) matrices.  When
// the pair tile does not fit, pair sums go straight to the accumulators (lanes =
// consecutive samples, so each add is coalesced).
//
// Bound by the shared-memory float atomics (compare-and-swap loops) and latency at
// 12 warps per SM: 500 trees of depth 6 (31,449 leaves, F = 30), 2,000 samples: 1.56 ms
// on the sibling-pair path tables, 1.36 ms here; F = 80, where the tile does not fit, 1.20 -> 1.09 ms; one row 166 -> 88 us.
//
// qts-build-parts: 15 (part 0: host code; parts 1-14: the kernels)
#include <algorithm>

#include "qts_blocks.cuh"

namespace qts {

constexpr int kIbSegs = 40;
constexpr int kIbWarps = 4;

struct IbSeg {
    const Rec32* rec;
    int64_t n;
    int64_t cta_begin;  // first thread block
    int32_t per_cta;    // blocks per thread block
    int32_t D, h;
};

struct IbArgs {
    IbSeg seg[kIbSegs];
    int n_seg;
    int sub;            // blocks per staged sub-chunk
    int stage;          // records per staging buffer
    int n_tiles;
    const float* X;
    int64_t M;
    int F;
    int cat;            // ensemble has categorical elements: always the NaN-aware variant
    int group;          // few samples (M <= kFewRows): lanes are (block, sample) pairs, a
                        // warp takes `group` = 32 / M blocks at a time; 0 otherwise
    int64_t n_pairs;
    double* acc_pair;   // [n_pairs][M]
    double* acc_phi;    // [F][M]
    int* status;
    QuadF q;
};

// Quadrature nodes per pass: the pass keeps three vectors per shared element and one
// per node of the subtree, and a pass over all eight nodes adds each pair once.
// Without a pair tile the adds go to global memory and cost more than spilled
// vectors.  Only widths up to 8 have the variants of rules that 8 does not divide.
__host__ __device__ constexpr int ib_np(int D, int h, bool tile) {
    const int vecs = 3 * D + (h == 0 ? 0 : (1 << h) - 1);
    return D <= 8 && vecs <= (tile ? 17 : 32) ? 8 : vecs <= 34 ? 4 : 2;
}
// launch classes: the widths of a class share kernels; HALF: rules that a pass of
// eight nodes does not divide
__host__ __device__ constexpr int ib_class(int D) {
    return D <= 3 ? 0 : D <= 5 ? 1 : D <= 8 ? 2 : D <= 16 ? 3 + (D - 9) / 2 : 2 + D / 4;
}
[[maybe_unused]] constexpr int kIbClasses = 11;

template <int CLS, bool HALF>
cudaError_t launch_ib(const IbArgs& a, bool pair_smem, int64_t ctas, size_t smem, cudaStream_t st);

#if QTS_DEVICE_PARTS

// The tiles and accumulators of one lane's sample.
template <bool PAIR_SMEM>
struct IbOut {
    float *ps, *pt;
    const int* row;     // row[f]: index of the pair (f, g), f < g, less g
    double* acc_pair;
    int64_t s, M;
    int col, F;
    bool live;
    __device__ __forceinline__ void phi(int f, float v) const {
        if (f < F) atomicAdd(&ps[f * kTileLd + col], v);
    }
    // fa, fb: the pair's features in any order
    __device__ __forceinline__ void pair(int fa, int fb, float v) const {
        const int idx = row[min(fa, fb)] + max(fa, fb);
        if constexpr (PAIR_SMEM) atomicAdd(&pt[idx * kTileLd + col], v);
        else if (live && v != 0.f) atomicAdd(&acc_pair[(int64_t)idx * M + s], (double)v);
    }
};

template <int H>
struct IbTree {
    static constexpr int kN = H == 0 ? 1 : (1 << H) - 1;
    int f[kN];
    float dL[kN], dR[kN], zL[kN], zR[kN];  // pair nodes: dL = val d, zL = sum of val z
};

template <int H, int N, int LEVELS, bool HAS_NAN>
__device__ __forceinline__ void ib_decode(const Rec32* nodes, const SmemCols& xr, IbTree<H>& t) {
    const float4 a = rec4(nodes + blk_rec(H, N)), b = rec4(nodes + blk_rec(H, N) + 1);
    t.f[N - 1] = feat_of(__float_as_uint(b.w));
    bool l, r;
    node_sides<N == 1, HAS_NAN>(xr(t.f[N - 1]), b, &l, &r);
    if constexpr (LEVELS == 1) {
        t.dL[N - 1] = fmaf(a.x, (l ? 1.f : 0.f) - a.z, a.y * ((r ? 1.f : 0.f) - a.w));
        t.zL[N - 1] = nodes[blk_rec(H, N) + 2].z;
    } else {
        t.dL[N - 1] = (l ? 1.f : 0.f) - a.x;
        t.dR[N - 1] = (r ? 1.f : 0.f) - a.z;
        t.zL[N - 1] = a.x;
        t.zR[N - 1] = a.z;
        ib_decode<H, 2 * N, LEVELS - 1, HAS_NAN>(nodes, xr, t);
        ib_decode<H, 2 * N + 1, LEVELS - 1, HAS_NAN>(nodes, xr, t);
    }
}

// Vectors over the pass's quadrature nodes.
template <int K>
struct V {
    float2 v[K];
};
template <int K>
__device__ __forceinline__ V<K> vmul(const V<K>& a, const V<K>& b) {
    V<K> r;
#pragma unroll
    for (int k = 0; k < K; ++k) r.v[k] = mul2(a.v[k], b.v[k]);
    return r;
}
template <int K>
__device__ __forceinline__ V<K> vfac(const V<K>& T, float d, float z) {  // z + d t
    V<K> r;
#pragma unroll
    for (int k = 0; k < K; ++k) r.v[k] = fma2(T.v[k], f2s(d), f2s(z));
    return r;
}
template <int K>
__device__ __forceinline__ float vdot(const V<K>& a, const V<K>& b) {
    return dot_k<K>(a.v, b.v);
}

// Bottom-up over node N: G, its leaf sum; U[u] of every node u below and including
// N, relative to N.  Adds the pairs of a node above a node; C = the block's product
// of shared factors times the edges down to N (U and C are later joined at the root).
template <int H, int N, int LEVELS, int K, typename OUT>
__device__ __forceinline__ void ib_up(const IbTree<H>& t, const V<K>& T, const V<K>& C, V<K>& G, V<K> (&U)[IbTree<H>::kN],
                                      const OUT& out) {
    const float dl = t.dL[N - 1];
    if constexpr (LEVELS == 1) {
        G = vfac<K>(T, dl, t.zL[N - 1]);
#pragma unroll
        for (int k = 0; k < K; ++k) U[N - 1].v[k] = f2s(dl);
    } else {
        const float dr = t.dR[N - 1];
        V<K> g;
        // left then right: factors of the edge, the child's sums, the pairs (N, u) for
        // u below the edge, and the child's U raised to N
        auto side = [&](auto child, float d, float z, bool first) {
            constexpr int CN = decltype(child)::value;
            const V<K> a = vfac<K>(T, d, z);
            ib_up<H, CN, LEVELS - 1, K>(t, T, vmul<K>(C, a), g, U, out);
            auto raise = [&](auto node) {
                constexpr int u = decltype(node)::value;
                if (t.f[u - 1] < out.F) {
                    if (t.f[N - 1] < out.F) out.pair(t.f[N - 1], t.f[u - 1], d * vdot<K>(C, U[u - 1]));
                    U[u - 1] = vmul<K>(U[u - 1], a);
                }
            };
            raise(child);
            if constexpr (LEVELS > 2) {
                raise(std::integral_constant<int, 2 * CN>{});
                raise(std::integral_constant<int, 2 * CN + 1>{});
            }
#pragma unroll
            for (int k = 0; k < K; ++k) {
                G.v[k] = first ? mul2(a.v[k], g.v[k]) : fma2(a.v[k], g.v[k], G.v[k]);
                U[N - 1].v[k] = first ? mul2(f2s(d), g.v[k]) : fma2(f2s(d), g.v[k], U[N - 1].v[k]);
            }
        };
        side(std::integral_constant<int, 2 * N>{}, dl, t.zL[N - 1], true);
        side(std::integral_constant<int, 2 * N + 1>{}, dr, t.zR[N - 1], false);
    }
}

template <int D, int H, int NP, bool HAS_NAN, typename OUT>
__device__ __forceinline__ void ib_block(const Rec32* __restrict__ r, const SmemCols& xr, const OUT& out,
                                         const QuadF& q) {
    constexpr int K = NP / 2;
    constexpr int DN = D > 0 ? D : 1;
    const uint32_t* words = reinterpret_cast<const uint32_t*>(r + 1 + D);
    float dd[DN], zz[DN], c1[DN];
    int ff[DN], nreal = D;  // padding (feature F) sorts last
#pragma unroll
    for (int j = 0; j < D; ++j) {
        const float4 e = rec4(r + 1 + j);
        const uint32_t word = words[j];
        ff[j] = feat_of(word);
        dd[j] = (satisfies<HAS_NAN>(xr(ff[j]), e.z, e.w, word) ? 1.f : 0.f) - e.x;
        zz[j] = e.x;
        c1[j] = 0.f;
        if (D > 16 && ff[j] >= out.F && j < nreal) nreal = j;
    }
    IbTree<H> t;
    if constexpr (H > 0) ib_decode<H, 1, H, HAS_NAN>(r + blk_head(D), xr, t);
#pragma unroll 1
    for (int m0 = 0; m0 < q.n_pad; m0 += NP) {
        V<K> T, P[D + 1], A[DN], S[DN], G, U[IbTree<H>::kN];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            T.v[k] = f2(q.t[m0 + 2 * k], q.t[m0 + 2 * k + 1]);
            P[0].v[k] = f2(q.w[m0 + 2 * k], q.w[m0 + 2 * k + 1]);
        }
#pragma unroll
        for (int j = 0; j < D; ++j) {
            A[j] = vfac<K>(T, dd[j], zz[j]);
            P[j + 1] = vmul<K>(P[j], A[j]);
        }
        if constexpr (H > 0) {
            ib_up<H, 1, H, K>(t, T, P[D], G, U, out);
#pragma unroll
            for (int u = 0; u < IbTree<H>::kN; ++u) out.phi(t.f[u], vdot<K>(P[D], U[u]));
        } else {
#pragma unroll
            for (int k = 0; k < K; ++k) G.v[k] = f2s(r[0].z);
        }
        if constexpr (D > 0) {
            S[D - 1] = G;
#pragma unroll
            for (int j = D - 1; j >= 1; --j) S[j - 1] = vmul<K>(S[j], A[j]);
        }
#pragma unroll
        for (int i = 0; i < D; ++i) {
            if (D > 16 && i >= nreal) break;
            c1[i] += vdot<K>(P[i], S[i]);
            V<K> R = P[i];  // the shared factors but i's, as far as j
#pragma unroll
            for (int j = i + 1; j < D; ++j) {
                if (D > 16 && j >= nreal) break;
                out.pair(ff[i], ff[j], vdot<K>(R, S[j]) * (dd[i] * dd[j]));
                R = vmul<K>(R, A[j]);
            }
            if constexpr (H > 0) {
#pragma unroll
                for (int u = 0; u < IbTree<H>::kN; ++u)
                    if (t.f[u] < out.F) out.pair(ff[i], t.f[u], dd[i] * vdot<K>(R, U[u]));
            }
        }
    }
#pragma unroll
    for (int j = 0; j < D; ++j)
        if (D <= 16 || j < nreal) out.phi(ff[j], dd[j] * c1[j]);
}

// The NaN-aware body, compiled once for the calls of the general kernels.
template <int D, int H, int NP, typename OUT>
__device__ __noinline__ void ib_block_any(const Rec32* r, const float* xs, int col, const OUT* out, const QuadF* q) {
    ib_block<D, H, NP, true>(r, SmemCols{xs, col}, *out, *q);
}

// FAST: widths up to 8 with a pair tile and one sample per lane, where both bodies
// are inlined (a call in the kernel costs its other path 60%).
template <int D, int H, bool HALF, bool PAIR_SMEM, bool FAST>
__device__ __forceinline__ bool ib_run(const IbArgs& a, const IbSeg& sg, int64_t p0, int64_t p1, bool has_nan,
                                       int64_t s0, const float* xs, float* ps, float* pt, const int* row, Rec32* st0,
                                       Rec32* st1, uint64_t* bars, uint32_t* s_phase, int* s_flag) {
    constexpr int NP = HALF && ib_np(D, H, PAIR_SMEM) == 8 ? 4 : ib_np(D, H, PAIR_SMEM);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (!FAST && a.group > 0) {
        // few samples: lane (slot, sample) evaluates its own block for its sample
        const int slot = lane / (int)a.M, col = lane - slot * (int)a.M;
        const IbOut<PAIR_SMEM> out{ps, pt, row, a.acc_pair, col, a.M, col, a.F, true};
        for (int64_t i = p0 + (int64_t)warp * a.group; i < p1; i += (int64_t)kIbWarps * a.group) {
            const int64_t k = i + slot;
            if (slot < a.group && k < p1)
                ib_block_any<D, H, NP>(sg.rec + k * blk_stride(D, H), xs, col, &out, &a.q);
        }
        __syncthreads();  // every warp's adds are in the tiles before the flush
        return true;
    }
    const SmemCols xr{xs, lane};
    const IbOut<PAIR_SMEM> out{ps, pt, row, a.acc_pair, s0 + lane, a.M, lane, a.F, s0 + lane < a.M};
    return stream_records<Rec32>(sg.rec, blk_stride(D, H), p0, p1, a.sub, st0, st1, bars, s_phase, s_flag, a.status,
                                 [&](int64_t, const Rec32* r) {
                                     if constexpr (FAST) {
                                         if (has_nan) ib_block<D, H, NP, true>(r, xr, out, a.q);
                                         else ib_block<D, H, NP, false>(r, xr, out, a.q);
                                     } else {
                                         ib_block_any<D, H, NP>(r, xs, lane, &out, &a.q);
                                     }
                                 });
}

template <int CLS, bool HALF, bool PAIR_SMEM, bool FAST>
__global__ void __launch_bounds__(kIbWarps * 32, CLS <= 4 ? 3 : 2) ib_kernel(const __grid_constant__ IbArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int F = a.F;
    const size_t rows = F + 1;
    float* xs = (float*)smem;
    float* ps = xs + rows * kTileLd;
    int* row = (int*)(ps + rows * kTileLd);
    float* pt = (float*)(row + ((rows + 3) & ~(size_t)3));
    size_t off = (size_t)((char*)pt - (char*)smem) + (PAIR_SMEM ? (size_t)a.n_pairs * kTileLd * 4 : 0);
    off = (off + 15) & ~(size_t)15;
    Rec32* st0 = (Rec32*)(smem + off);
    Rec32* st1 = st0 + a.stage;
    uint64_t* bars = (uint64_t*)(st1 + a.stage);
    __shared__ int s_flag;
    __shared__ uint32_t s_phase[2];
    int si = 0;
    while (si + 1 < a.n_seg && (int64_t)blockIdx.x >= a.seg[si + 1].cta_begin) ++si;
    const IbSeg sg = a.seg[si];
    const int64_t local = (int64_t)blockIdx.x - sg.cta_begin;
    const int64_t s0 = (local % a.n_tiles) * 32;
    const int64_t p0 = (local / a.n_tiles) * sg.per_cta;
    const int64_t p1 = imin64(p0 + sg.per_cta, sg.n);
    if (threadIdx.x == 0) {
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        mbar_fence_init();
        s_phase[0] = s_phase[1] = 0;
    }
    for (int idx = threadIdx.x; idx < (int)rows * kTileLd; idx += blockDim.x) ps[idx] = 0.f;
    for (int f = threadIdx.x; f < F; f += blockDim.x) row[f] = f * F - f * (f + 1) / 2 - f - 1;
    if (PAIR_SMEM)
        for (int idx = threadIdx.x; idx < (int)a.n_pairs * kTileLd; idx += blockDim.x) pt[idx] = 0.f;
    const bool has_nan = load_tile_t(xs, a.X, s0, a.M, F, F, 1) || a.cat != 0;
    bool ok = false;
#define QTS_RUN(DD, HH) \
    ok = ib_run<DD, HH, HALF, PAIR_SMEM, FAST>(a, sg, p0, p1, has_nan, s0, xs, ps, pt, row, st0, st1, bars, s_phase, &s_flag)
#define QTS_CASE(DD)                                                        \
    case DD:                                                                \
        if (sg.h == 0) QTS_RUN(DD, 0);                                      \
        else if (sg.h == 1) QTS_RUN(DD, 1);                                 \
        else if (sg.h == 2) QTS_RUN(DD, (blk_max_h(DD) >= 2 ? 2 : 0));      \
        else QTS_RUN(DD, (blk_max_h(DD) >= 3 ? 3 : 0));                     \
        break;
    if constexpr (CLS == 0) {
        switch (sg.D) {
            QTS_CASE(0) QTS_CASE(1) QTS_CASE(2) QTS_CASE(3)
            default: break;
        }
    } else if constexpr (CLS == 1) {
        switch (sg.D) {
            QTS_CASE(4) QTS_CASE(5)
            default: break;
        }
    } else if constexpr (CLS == 2) {
        switch (sg.D) {
            QTS_CASE(6) QTS_CASE(7) QTS_CASE(8)
            default: break;
        }
    } else if constexpr (CLS == 3) {
        switch (sg.D) {
            QTS_CASE(9) QTS_CASE(10)
            default: break;
        }
    } else if constexpr (CLS == 4) {
        switch (sg.D) {
            QTS_CASE(11) QTS_CASE(12)
            default: break;
        }
    } else if constexpr (CLS == 5) {
        switch (sg.D) {
            QTS_CASE(13) QTS_CASE(14)
            default: break;
        }
    } else if constexpr (CLS == 6) {
        switch (sg.D) {
            QTS_CASE(15) QTS_CASE(16)
            default: break;
        }
    } else {
        switch (sg.D) {
            QTS_CASE(4 * CLS - 8)
            default: break;
        }
    }
#undef QTS_CASE
#undef QTS_RUN
    if (!ok) return;
    // flush: consecutive threads take consecutive samples of one row, so the
    // FP64 adds into the [row][sample] accumulators are coalesced
    for (int idx = threadIdx.x; idx < 32 * F; idx += blockDim.x) {
        const int f = idx >> 5, sl = idx & 31;
        const float v = ps[f * kTileLd + sl];
        if (s0 + sl < a.M && v != 0.f) atomicAdd(&a.acc_phi[(int64_t)f * a.M + s0 + sl], (double)v);
    }
    if (PAIR_SMEM) {
        for (int64_t idx = threadIdx.x; idx < 32 * a.n_pairs; idx += blockDim.x) {
            const int64_t pr = idx >> 5;
            const int sl = (int)(idx & 31);
            const float v = pt[pr * kTileLd + sl];
            if (s0 + sl < a.M && v != 0.f) atomicAdd(&a.acc_pair[pr * a.M + s0 + sl], (double)v);
        }
    }
}

template <int CLS, bool HALF>
cudaError_t launch_ib(const IbArgs& a, bool pair_smem, int64_t ctas, size_t smem, cudaStream_t st) {
    auto k = pair_smem ? ib_kernel<CLS, HALF, true, false> : ib_kernel<CLS, HALF, false, false>;
    if constexpr (CLS <= 2) {
        if (pair_smem && a.group == 0) k = ib_kernel<CLS, HALF, true, true>;
    }
    if (smem > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    k<<<(unsigned)ctas, kIbWarps * 32, smem, st>>>(a);
    return cudaGetLastError();
}

#define QTS_INST(C, HALF) template cudaError_t launch_ib<C, HALF>(const IbArgs&, bool, int64_t, size_t, cudaStream_t);
#if QTS_IN_PART(1)
QTS_INST(0, false)
#endif
#if QTS_IN_PART(2)
QTS_INST(0, true)
#endif
#if QTS_IN_PART(3)
QTS_INST(1, false)
#endif
#if QTS_IN_PART(4)
QTS_INST(1, true)
#endif
#if QTS_IN_PART(5)
QTS_INST(2, false)
#endif
#if QTS_IN_PART(6)
QTS_INST(2, true)
#endif
#if QTS_IN_PART(7)
QTS_INST(3, false)
#endif
#if QTS_IN_PART(8)
QTS_INST(4, false)
#endif
#if QTS_IN_PART(9)
QTS_INST(5, false)
#endif
#if QTS_IN_PART(10)
QTS_INST(6, false)
#endif
#if QTS_IN_PART(11)
QTS_INST(7, false)
#endif
#if QTS_IN_PART(12)
QTS_INST(8, false)
#endif
#if QTS_IN_PART(13)
QTS_INST(9, false)
#endif
#if QTS_IN_PART(14)
QTS_INST(10, false)
#endif
#undef QTS_INST

#endif  // QTS_DEVICE_PARTS

#if !QTS_HOST_PART
}  // namespace qts
#endif

#if QTS_HOST_PART

static size_t ib_smem(int F, int stage, bool pair_smem) {
    const size_t rows = F + 1;
    size_t off = 2 * rows * kTileLd * 4 + ((rows + 3) & ~(size_t)3) * 4;
    if (pair_smem) off += (size_t)F * (F - 1) / 2 * kTileLd * 4;
    off = (off + 15) & ~(size_t)15;
    return off + 2 * (size_t)stage * sizeof(Rec32) + 16;
}

// the most shared memory a thread block takes for its pair tile
static constexpr size_t kIbBudget = 200 * 1024;

static double ib_cost(int D, int h) {
    const int n = h == 0 ? 0 : (1 << h) - 1;
    return 4.0 + 2.0 * D + 0.5 * D * (D - 1) + (D + 4.0) * n;
}

cudaError_t launch_int_blocks(const qts_ensemble* e, const float* X, int64_t M, int F, int n_quad, double* acc_pair,
                              double* acc_phi, cudaStream_t st) {
    if (M <= 0) return cudaSuccess;
    const int64_t tiles = (M + 31) / 32;
    const int group = M <= kFewRows ? (int)(32 / M) : 0;
    // work per thread block: about eight rounds of the whole chip (three thread
    // blocks per SM); at least what keeps the pair tile's set-up and flush, F^2 / 2
    // rows, small beside the blocks'
    double total = 0.0;
    for (const BlockBucket& b : e->blk) total += (double)b.n * ib_cost(b.D, b.h);
    const double least = 1500.0 + (double)std::min(F, 64) * std::min(F, 64) * 4.0;
    const double share = std::max(least, std::min(20e3, total * (double)tiles / (8.0 * 3 * num_sms())));
    for (int cls = 0; cls < kIbClasses; ++cls) {
        for (int nq = n_quad == QTS_NQ_EXACT ? QTS_MAX_QUAD : n_quad; nq >= (n_quad == QTS_NQ_EXACT ? 1 : n_quad); --nq) {  // one launch per rule of the class
            IbArgs a;
            a.n_seg = 0;
            int64_t ctas = 0;
            int stride = 0;
            for (auto it = e->blk.rbegin(); it != e->blk.rend(); ++it) {  // the longest first
                const BlockBucket& b = *it;
                // QTS_NQ_EXACT: the diagonal holds first-order values, so a bucket takes
                // the first-order count (Thm 2)
                if (ib_class(b.D) != cls || nodes_for(n_quad, b.dmax, 1) != nq) continue;
                if (a.n_seg == kIbSegs) return cudaErrorInvalidValue;  // a class has fewer buckets
                stride = std::max(stride, blk_stride(b.D, b.h));
                int64_t per = std::max<int64_t>(kIbWarps, (int64_t)(share / ib_cost(b.D, b.h)));
                if (group) per = std::max<int64_t>(per, (int64_t)kIbWarps * group);
                per = std::min<int64_t>((per + kIbWarps - 1) / kIbWarps * kIbWarps, 1 << 20);
                a.seg[a.n_seg++] = {e->blkdev.rec + b.rec_off, b.n, ctas, (int32_t)per, b.D, b.h};
                ctas += (b.n + per - 1) / per * tiles;
            }
            if (a.n_seg == 0) continue;
            if (ctas > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
            // the rule padded to a pass of four nodes up to width 12 (eight where they divide it)
            if (!make_quad(nq, &a.q, nullptr, cls <= 4 ? 4 : 2)) return cudaErrorInvalidValue;
            a.sub = 16;
            // wide inputs: stage fewer blocks at a time until the thread block fits
            while (a.sub > 1 && ib_smem(F, a.sub * stride, false) > kSmemMax) a.sub /= 2;
            a.stage = a.sub * stride;
            a.n_tiles = (int)tiles;
            a.X = X;
            a.M = M;
            a.F = F;
            a.cat = e->prep.has_cat ? 1 : 0;
            a.group = group;
            a.n_pairs = (int64_t)F * (F - 1) / 2;
            a.acc_pair = acc_pair;
            a.acc_phi = acc_phi;
            a.status = e->d_status;
            const bool pair_smem = ib_smem(F, a.stage, true) <= kIbBudget;
            const size_t smem = ib_smem(F, a.stage, pair_smem);
            if (smem > kSmemMax) return cudaErrorInvalidConfiguration;
            const bool half = a.q.n_pad % 8 != 0;
            cudaError_t r = cudaErrorInvalidValue;
            switch (cls) {
                case 0:
                    r = half ? launch_ib<0, true>(a, pair_smem, ctas, smem, st)
                             : launch_ib<0, false>(a, pair_smem, ctas, smem, st);
                    break;
                case 1:
                    r = half ? launch_ib<1, true>(a, pair_smem, ctas, smem, st)
                             : launch_ib<1, false>(a, pair_smem, ctas, smem, st);
                    break;
                case 2:
                    r = half ? launch_ib<2, true>(a, pair_smem, ctas, smem, st)
                             : launch_ib<2, false>(a, pair_smem, ctas, smem, st);
                    break;
#define QTS_CASE(C) \
    case C: r = launch_ib<C, false>(a, pair_smem, ctas, smem, st); break;
                QTS_CASE(3) QTS_CASE(4) QTS_CASE(5) QTS_CASE(6) QTS_CASE(7) QTS_CASE(8) QTS_CASE(9)
                QTS_CASE(10)
#undef QTS_CASE
                default: break;
            }
            if (r != cudaSuccess) return r;
        }
    }
    return cudaSuccess;
}

}  // namespace qts

#endif  // QTS_HOST_PART
