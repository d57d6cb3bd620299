// Adjoint of the first-order path (the paper has no adjoint; this
// differentiates Thm 1 / Eq. shap_as_weighted_banzhafs with the same n-point
// rule).  With L = sum_s sum_f grad_phi[s,f] phi[s,f], g_j = grad_phi[s, f_j],
// d_j = o_j - z_j, u_j = g_j d_j and a_j(t) = z_j + t d_j:
//
//   dL/dval   = sum_s sum_m w_m sum_i u_i prod_{l != i} a_l(t_m)
//   dL/dz_k   = sum_s val sum_m w_m [ -g_k prod_{l != k} a_l
//                                     + (1 - t_m) sum_{i != k} u_i prod_{l not in {i,k}} a_l ]
//
// (plus the bias terms of E[f], added in the epilogue).  Both are O(d) per
// (sample, path, node) with dual prefix products P_j = prod_{l<j} a_l,
// PU_j = sum_{i<j} u_i prod_{l<j, l != i} a_l and the matching suffixes S, SU:
//   prod_{l != k} a_l = P_k S_k,   sum_{i != k} u_i prod_{l != i,k} a_l = PU_k S_k + P_k SU_k.
// Products are recomputed per call, never stored.  An epilogue chains the
// elements' gradients to the tree's edges:
// dL/dw_e = dL/dz_k * prod_{other edges e' merged into k} w_e'.
//
// FP32 runs on the block tables with the batched pass's kernels (qts_batch.cu);
// this file holds the FP64 kernels, which run path by path:
// lanes are samples, the per-path sums over a tile of 32 samples are reduced in
// the warp and added to FP64 per-path / per-element accumulators.
//
// qts-build-parts: 6 (part 0: host code; parts 1-5: the per-width kernels)
#include <algorithm>
#include <type_traits>

#include "qts_paths.cuh"

namespace qts {

struct BwdArgs {
    const void* rec;
    int64_t n_paths;
    int64_t paths_per_block;
    int sub;
    int n_tiles;
    const float* X;
    const float* G;     // grad_phi, M x (F+1)
    int64_t M;
    int F;
    int cat;            // ensemble has categorical elements: always the NaN-aware variant
    double* g_val;      // per path of this bucket
    double* g_slot;     // per element slot of this bucket (n_paths * D)
    int* status;
    QuadD qd;
};

template <int D>
cudaError_t launch_bwd_d(const BwdArgs& a, int warps, int64_t blocks, size_t smem, cudaStream_t st);

#if QTS_DEVICE_PARTS

// --------------------------------------------------------------- kernel ---

__device__ __forceinline__ void bwd_smem_layout(int F, int sub, int D, float** xs, float** gs, Rec64** st0, Rec64** st1,
                                                uint64_t** bars, unsigned char* base) {
    const size_t rows = F + 1;
    size_t off = 0;
    *xs = (float*)(base + off);
    off += rows * kTileLd * sizeof(float);
    *gs = (float*)(base + off);
    off += rows * kTileLd * sizeof(float);
    off = (off + 15) & ~(size_t)15;
    *st0 = (Rec64*)(base + off);
    off += (size_t)sub * (D + 1) * sizeof(Rec64);
    *st1 = (Rec64*)(base + off);
    off += (size_t)sub * (D + 1) * sizeof(Rec64);
    off = (off + 15) & ~(size_t)15;
    *bars = (uint64_t*)(base + off);
}

template <int D>
__global__ void __launch_bounds__(256) bwd_kernel(BwdArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    float *xs, *gs;
    Rec64 *st0, *st1;
    uint64_t* bars;
    bwd_smem_layout(a.F, a.sub, D, &xs, &gs, &st0, &st1, &bars, smem);
    __shared__ int s_flag;
    __shared__ uint32_t s_phase[2];

    const int F = a.F;
    const int lane = threadIdx.x & 31;
    const int tile = (int)(blockIdx.x % (unsigned)a.n_tiles);
    const int64_t chunk = blockIdx.x / (unsigned)a.n_tiles;
    const int64_t s0 = (int64_t)tile * 32;
    const int64_t p0 = chunk * a.paths_per_block;
    const int64_t p1 = imin64(p0 + a.paths_per_block, a.n_paths);

    if (threadIdx.x == 0) {
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        mbar_fence_init();
        s_phase[0] = s_phase[1] = 0;
    }
    const bool has_nan = load_tile_t(xs, a.X, s0, a.M, F, F, 1) || a.cat != 0;
    // grad_phi tile: columns 0..F-1 (column F, the bias weight, is handled in
    // the epilogue); row F stays zero for padding elements
    load_tile_t(gs, a.G, s0, a.M, F, F + 1, 1);

    (void)stream_paths<Rec64, D>(
        (const Rec64*)a.rec, p0, p1, a.sub, st0, st1, bars, s_phase, &s_flag, a.status,
        [&](int64_t p, const Rec64* r) {
            double* gsl = a.g_slot + p * D;
            double* gv = a.g_val + p;
            if (has_nan) bwd_path_f64<D, true>(r, xs, gs, lane, a.qd, gsl, gv);
            else bwd_path_f64<D, false>(r, xs, gs, lane, a.qd, gsl, gv);
        });
}

// ---------------------------------------------------------- launchers -----

template <int D>
cudaError_t launch_bwd_d(const BwdArgs& a, int warps, int64_t blocks, size_t smem, cudaStream_t st) {
    auto k = bwd_kernel<D>;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    k<<<(unsigned)blocks, warps * 32, smem, st>>>(a);
    return cudaGetLastError();
}

#define QTS_INST(DD) \
    template cudaError_t launch_bwd_d<DD>(const BwdArgs&, int, int64_t, size_t, cudaStream_t);
#if QTS_IN_PART(1)
QTS_INST(64)
#endif
#if QTS_IN_PART(2)
QTS_INST(56)
#endif
#if QTS_IN_PART(3)
QTS_INST(48) QTS_INST(40)
#endif
#if QTS_IN_PART(4)
QTS_INST(32) QTS_INST(28) QTS_INST(24) QTS_INST(20)
#endif
#if QTS_IN_PART(5)
QTS_INST(1) QTS_INST(2) QTS_INST(3) QTS_INST(4) QTS_INST(5) QTS_INST(6) QTS_INST(7) QTS_INST(8) QTS_INST(9) QTS_INST(10) QTS_INST(11) QTS_INST(12) QTS_INST(13) QTS_INST(14) QTS_INST(15) QTS_INST(16)
#endif
#undef QTS_INST

#endif  // QTS_DEVICE_PARTS

#if !QTS_HOST_PART
}  // namespace qts
#endif

#if QTS_HOST_PART

size_t bwd_smem_bytes(int F, int sub, int D) {
    size_t off = 2 * (size_t)(F + 1) * kTileLd * 4;
    off = (off + 15) & ~(size_t)15;
    off += 2 * (size_t)sub * (D + 1) * sizeof(Rec64);
    off = (off + 15) & ~(size_t)15;
    return off + 16;
}

// ------------------------------------------------------------ epilogue ----

// G = sum_s grad_phi[s, F]  (the weight of E[f] in L), FP64.
__global__ void bias_grad_kernel(const float* __restrict__ G, int64_t M, int F, double* out) {
    double acc = 0.0;
    for (int64_t s = threadIdx.x; s < M; s += blockDim.x) acc += (double)G[s * (F + 1) + F];
    for (int off = 16; off >= 1; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    __shared__ double part[32];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += part[w];
        *out = t;
    }
}

// d_leaf of every path's leaf: sum over samples + bias term G * prod_j z_j;
// single-leaf trees contribute G (their value is part of E[f] directly).
__global__ void path_epilogue_kernel(int64_t n_paths, const int64_t* __restrict__ leaf,
                                     const double* __restrict__ zprod, const double* __restrict__ g_val,
                                     const double* __restrict__ gb, int64_t n_empty,
                                     const int64_t* __restrict__ empty_leaf, double* d_leaf) {
    const double G = *gb;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n_paths + n_empty;
         p += (int64_t)gridDim.x * blockDim.x) {
        if (p < n_paths) d_leaf[leaf[p]] = g_val[p] + G * zprod[p];
        else d_leaf[empty_leaf[p - n_paths]] = G;
    }
}

struct SlotMap {
    int nb;
    int64_t slot_base[kMaxBuckets + 1];
    int64_t path_base[kMaxBuckets];
    int D[kMaxBuckets];
};

// Chain each element's dL/dz to the edges merged into it.
__global__ void slot_epilogue_kernel(SlotMap sm, const double* __restrict__ g_slot,
                                     const double* __restrict__ path_val,
                                     const double* __restrict__ zexcl, const int64_t* __restrict__ eb,
                                     const int64_t* __restrict__ enode, const double* __restrict__ ecoef,
                                     const double* __restrict__ gb, double* d_z) {
    const double G = *gb;
    const int64_t n_slots = sm.slot_base[sm.nb];
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n_slots;
         s += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e0 = eb[s], e1 = eb[s + 1];
        if (e0 == e1) continue;  // padding slot
        int b = 0;
        while (b + 1 < sm.nb && s >= sm.slot_base[b + 1]) ++b;
        const int64_t p = sm.path_base[b] + (s - sm.slot_base[b]) / sm.D[b];
        const double tot = g_slot[s] + G * path_val[p] * zexcl[s];
        for (int64_t e = e0; e < e1; ++e) atomicAdd(&d_z[enode[e]], tot * ecoef[e]);
    }
}

// FP64, on the per-leaf tables
static cudaError_t launch_bwd_bucket(const qts_ensemble* e, const Bucket& b, const float* X, const float* grad,
                                     int64_t M, int F, const QuadD& qd, double* g_val, double* g_slot,
                                     const Tune& tn, cudaStream_t st) {
    if (M <= 0 || b.n_paths == 0) return cudaSuccess;
    BwdArgs a;
    a.rec = (const Rec64*)e->d_rec + b.rec_off;
    a.n_paths = b.n_paths;
    a.sub = std::max(1, tn.sub);
    // wide inputs: stage fewer paths at a time until the block fits shared memory
    while (a.sub > 1 && bwd_smem_bytes(F, a.sub, b.D) > kSmemMax) a.sub /= 2;
    a.paths_per_block = std::max<int64_t>(a.sub, (int64_t)tn.paths / a.sub * a.sub);
    a.n_tiles = (int)((M + 31) / 32);
    a.X = X;
    a.G = grad;
    a.M = M;
    a.F = F;
    a.cat = e->prep.has_cat ? 1 : 0;
    a.g_val = g_val + b.path_base;
    a.g_slot = g_slot + b.slot_base;
    a.status = e->d_status;
    a.qd = qd;
    const int64_t chunks = (b.n_paths + a.paths_per_block - 1) / a.paths_per_block;
    const int64_t blocks = chunks * a.n_tiles;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    const size_t smem = bwd_smem_bytes(F, a.sub, b.D);
    if (smem > kSmemMax) return cudaErrorInvalidConfiguration;
    const int warps = std::max(1, std::min(8, tn.warps));
    switch (b.D) {
#define QTS_CASE(DD) \
    case DD: return launch_bwd_d<DD>(a, warps, blocks, smem, st);
        QTS_CASE(1) QTS_CASE(2) QTS_CASE(3) QTS_CASE(4) QTS_CASE(5) QTS_CASE(6) QTS_CASE(7)
        QTS_CASE(8) QTS_CASE(9) QTS_CASE(10) QTS_CASE(11) QTS_CASE(12) QTS_CASE(13) QTS_CASE(14)
        QTS_CASE(15) QTS_CASE(16) QTS_CASE(20) QTS_CASE(24) QTS_CASE(28) QTS_CASE(32)
        QTS_CASE(40) QTS_CASE(48) QTS_CASE(56) QTS_CASE(64)
#undef QTS_CASE
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_bwd_epilogue(const qts_ensemble* e, const float* grad, int64_t M, int F,
                                const double* g_val, const double* g_slot, double* d_leaf,
                                double* d_z, double* gb, cudaStream_t st) {
    const Prepared& P = e->prep;
    cudaError_t err = cudaMemsetAsync(d_leaf, 0, sizeof(double) * e->n_nodes, st);
    if (err == cudaSuccess) err = cudaMemsetAsync(d_z, 0, sizeof(double) * e->n_nodes, st);
    if (err != cudaSuccess) return err;
    bias_grad_kernel<<<1, 1024, 0, st>>>(grad, M, F, gb);
    const int64_t np = P.n_paths + (int64_t)P.empty_leaf.size();
    if (np > 0) {
        const int blocks = (int)std::min<int64_t>((np + 255) / 256, 8 * 152);
        path_epilogue_kernel<<<blocks, 256, 0, st>>>(P.n_paths, e->d_path_leaf, e->d_path_zprod,
                                                     g_val, gb, (int64_t)P.empty_leaf.size(),
                                                     e->d_empty_leaf, d_leaf);
    }
    if (P.n_slots > 0) {
        SlotMap sm;
        sm.nb = (int)P.buckets.size();
        for (int b = 0; b < sm.nb; ++b) {
            sm.slot_base[b] = P.buckets[b].slot_base;
            sm.path_base[b] = P.buckets[b].path_base;
            sm.D[b] = P.buckets[b].D;
        }
        sm.slot_base[sm.nb] = P.n_slots;
        const int blocks = (int)std::min<int64_t>((P.n_slots + 255) / 256, 8 * 152);
        slot_epilogue_kernel<<<blocks, 256, 0, st>>>(sm, g_slot, e->d_path_val, e->d_slot_zexcl,
                                                     e->d_slot_edge_begin, e->d_edge_node,
                                                     e->d_edge_coef, gb, d_z);
    }
    return cudaGetLastError();
}

}  // namespace qts

using namespace qts;

extern "C" qts_status qts_shap_backward(qts_ensemble* e, const float* X, int64_t M, int32_t F,
                                        int32_t n_quad, const float* grad_phi, double* d_leaf,
                                        double* d_z, qts_stream_t stream) try {
    qts_status st = check_call(e, X, M, F, n_quad);
    if (st != QTS_OK) return st;
    if (!d_leaf || !d_z) return fail(QTS_ERR_ARG, "d_leaf and d_z must be non-NULL");
    if (M > 0 && !grad_phi) return fail(QTS_ERR_ARG, "grad_phi is NULL");
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t ce = cudaSuccess;
    if (M == 0) {
        ce = cudaMemsetAsync(d_leaf, 0, sizeof(double) * e->n_nodes, s);
        if (ce == cudaSuccess) ce = cudaMemsetAsync(d_z, 0, sizeof(double) * e->n_nodes, s);
        if (ce != cudaSuccess) return cuda_fail(ce, "adjoint epilogue");
        return QTS_OK;
    }
    if (!(e->flags & QTS_FLAG_FP64)) {
        // FP32: the block tables and the batched pass's kernels
        st = ensure_blocks(e, true);
        if (st != QTS_OK) return st;
        // The workspace holds a slab of the samples' transposed copies.  A stream
        // capture must not grow it: there a call that needs more takes memory of
        // the captured graph's own.
        int64_t slab = adjoint_slab(M, F);
        const size_t need = adjoint_work_bytes(e, slab, F);
        void* own = nullptr;
        if (need > e->work_bytes && is_capturing(s)) {
            ce = cudaMallocAsync(&own, need, s);
            if (ce != cudaSuccess) return cuda_fail(ce, "adjoint workspace");
        } else {
            st = ensure_workspace(e, need, s);
            // a device that is nearly full: smaller slabs
            for (int64_t k = smaller_slab(slab); st == QTS_ERR_OOM && k > 0; k = smaller_slab(k)) {
                slab = k;
                st = ensure_workspace(e, adjoint_work_bytes(e, slab, F), s);
            }
            if (st != QTS_OK) return st;
        }
        ce = launch_adjoint_blocks(e, own ? own : e->d_work, slab, X, grad_phi, M, F, n_quad, d_leaf, d_z, s);
        if (own) {
            const cudaError_t fe = cudaFreeAsync(own, s);
            if (ce == cudaSuccess) ce = fe;
        }
        return ce == cudaSuccess ? QTS_OK : cuda_fail(ce, "adjoint kernel launch");
    }
    const Prepared& P = e->prep;
    const size_t bytes = sizeof(double) * (size_t)(4 + P.n_paths + P.n_slots);
    st = ensure_workspace(e, bytes, s);
    if (st != QTS_OK) return st;
    double* gb = (double*)e->d_work;
    double* g_val = gb + 4;
    double* g_slot = g_val + P.n_paths;
    ce = cudaMemsetAsync(e->d_work, 0, bytes, s);
    if (ce != cudaSuccess) return cuda_fail(ce, "workspace clear");
    for (const Bucket& b : P.buckets) {
        // the bucket's rule (QTS_NQ_EXACT: ceil(D/2) points)
        QuadD qd;
        if (!make_quad(nodes_for(n_quad, b.D, 1), nullptr, &qd, 2)) return fail(QTS_ERR_ARG, "quadrature rule");
        ce = launch_bwd_bucket(e, b, X, grad_phi, M, F, qd, g_val, g_slot, e->tune[b.D], s);
        if (ce != cudaSuccess) return cuda_fail(ce, "adjoint kernel launch");
    }
    ce = launch_bwd_epilogue(e, grad_phi, M, F, g_val, g_slot, d_leaf, d_z, gb, s);
    if (ce != cudaSuccess) return cuda_fail(ce, "adjoint epilogue");
    return QTS_OK;
} QTS_ENTRY_END

#endif  // QTS_HOST_PART
