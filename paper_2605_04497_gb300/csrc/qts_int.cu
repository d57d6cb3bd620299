// Pairwise Shapley interaction values (Thm 1 with S = {i, j}; Alg. 1 with
// s = 2), in the pred_interactions layout: the entry points, the finalize kernel,
// and the kernels on path tables.  qts_shap_interactions runs on the block tables
// (qts_int_blocks.cu), or here with sibling leaves merged (pairs_on_paths); the
// allocation-free call may not build tables and runs here on the per-leaf ones.
//
// For a path with merged elements sorted by feature and a sample,
//     SII_ij += val d_i d_j sum_m w_m prod_{k != i,j} a_k(t_m),   d = o - z,
// computed without division: for each i the running product
// R = P_i * prod_{i<k<j} a_k (P_i = w_m val prod_{k<i} a_k) is extended one
// element at a time and multiplied by the stored suffix S_j = prod_{k>j} a_k.
// This is not a dense contraction (per path a rank-n_quad sum scattered over
// F^2/2 pair slots at density d/F), so it runs on the FP32 pipes, two nodes per
// f32x2 register pair.  Per block (32 samples x a chunk of paths) pair sums
// and first-order sums are accumulated in shared FP32 tiles and flushed into
// FP64 accumulators in the workspace laid out [pair][sample] and
// [feature][sample]; a finalize kernel writes the (F+1) x (F+1) matrices.
//
// All widths of a register class and rule are one launch (a thread block finds
// its segment by its index, and its paths follow from the call's work: one
// launch per width of 512 paths per thread block left most SMs idle on narrow
// widths; 500 trees of depth 6, 2,000 samples: 1.79 -> 1.56 ms).
//
// qts-build-parts: 7 (part 0: host code; parts 1-6: the kernels)
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

#include "qts_device.cuh"

namespace qts {

// Upper-triangle index of the pair (a, b), a < b < F.
__host__ __device__ __forceinline__ int64_t tri_index(int a, int b, int F) {
    return (int64_t)a * F - (int64_t)a * (a + 1) / 2 + (b - a - 1);
}

constexpr int kIntSegs = 24;
constexpr int kIntWarps = 4;

struct IntSeg {
    const Rec32* rec;
    int64_t n_paths;
    int64_t cta_begin;  // first thread block
    int32_t per_cta;    // paths per thread block
    int32_t D;
};

struct IntArgs {
    IntSeg seg[kIntSegs];
    int n_seg;
    int sub;            // paths per staged sub-chunk
    int stage;          // records per staging buffer
    int n_tiles;
    const float* X;
    int64_t M;
    int F;
    int cat;            // ensemble has categorical elements: always the NaN-aware variant
    int64_t n_pairs;
    int group;          // few samples (M <= 16): lanes are (path, sample) pairs, a warp
                        // takes `group` = 32 / M paths at a time; 0 otherwise
    double* acc_pair;   // [n_pairs][M]
    double* acc_phi;    // [F][M]
    int* status;
    QuadF q;
};

// the widest register pass a width takes (nodes per pass)
__host__ __device__ constexpr int int_max_np(int D) { return D <= 6 ? 8 : (D <= 12 ? 4 : 2); }

// launch classes: widths up to 4, 6, 8, 12, 16 and the padded ones above (7 and 8 with
// 9 to 12 held 155 registers instead of 109: 100 trees of depth 8, F = 56,
// 2,000 samples 2,879 instead of 2,260 us)
__host__ __device__ constexpr int int_class(int D) {
    return D <= 4 ? 0 : D <= 6 ? 1 : D <= 8 ? 2 : D <= 12 ? 3 : D <= 16 ? 4 : 5;
}
[[maybe_unused]] constexpr int kIntClasses = 6;

template <int CLS>
cudaError_t launch_int_c(const IntArgs& a, int np, bool pair_smem, int64_t blocks, size_t smem, cudaStream_t st);

#if QTS_DEVICE_PARTS

// d of a sibling pair's element (Rec32): the leaf that x reaches, or neither
template <bool HAS_NAN>
__device__ __forceinline__ float pair_d(float x, const Rec32& e, const Rec32& head) {
    bool in = x >= e.lo && x < e.hi, left = x < __uint_as_float(head.bits);
    if (HAS_NAN && x != x) {
        in = (e.bits & kNanOk) != 0;
        left = (e.bits & kDefLeft) != 0;
    }
    return !in ? -e.z : left ? head.lo : head.hi;
}

// PAIR_SMEM: pair sums go to a shared tile [n_pairs][33]; otherwise straight to
// the FP64 accumulator (lanes = consecutive samples, so each add is coalesced).
template <int D, int NP, bool HAS_NAN, bool PAIR_SMEM>
__device__ __forceinline__ void int_path_f32(const Rec32* __restrict__ r, const float* __restrict__ xs,
                                             float* ps, float* pt, double* acc_pair, int64_t s,
                                             int64_t M, int lane, int F, const QuadF& q) {
    constexpr int K = NP / 2;
    const float val = r[0].z;
    // a sibling pair (tables that merge them; they serve only calls without a pair
    // tile): its element sits last, after the padding and out of feature order,
    // and its two-leaf polynomial is one more linear factor of every term (val = 1)
    const bool pair = !PAIR_SMEM && (r[D].bits & kPairElem) != 0;
    float dd[D], c1[D];
    int nreal = D;  // sorted elements before the padding (padding sorts last)
#pragma unroll
    for (int j = 0; j < D; ++j) {
        const Rec32 e = r[1 + j];
        const int f = feat_of(e.bits);
        const float x = xs[f * kTileLd + lane];
        const bool o = satisfies<HAS_NAN>(x, e.lo, e.hi, e.bits);
        dd[j] = (o ? 1.f : 0.f) - e.z;
        if (j == D - 1 && pair) dd[j] = pair_d<HAS_NAN>(x, e, r[0]);
        c1[j] = 0.f;
        if (f >= F && j < nreal) nreal = j;
    }
    if (pair && nreal > D - 1) nreal = D - 1;
    const int npass = q.n_pad / NP;
    for (int pass = 0; pass < npass; ++pass) {
        float2 T[K], A[D][K], P[D][K], S[D][K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int m = pass * NP + 2 * k;
            T[k] = f2(q.t[m], q.t[m + 1]);
            P[0][k] = f2(q.w[m] * val, q.w[m + 1] * val);
        }
#pragma unroll
        for (int j = 0; j < D; ++j) {
            const float2 z2 = f2s(r[1 + j].z), d2 = f2s(dd[j]);
#pragma unroll
            for (int k = 0; k < K; ++k) {
                A[j][k] = fma2(T[k], d2, z2);
                if (j + 1 < D) P[j + 1][k] = mul2(P[j][k], A[j][k]);
            }
        }
#pragma unroll
        for (int k = 0; k < K; ++k) S[D - 1][k] = f2s(1.f);
#pragma unroll
        for (int j = D - 1; j >= 1; --j)
#pragma unroll
            for (int k = 0; k < K; ++k) S[j - 1][k] = mul2(S[j][k], A[j][k]);
        // first order: c1_j += sum_m P_j S_j
#pragma unroll
        for (int j = 0; j < D; ++j) {
            float2 a1 = mul2(P[j][0], S[j][0]);
#pragma unroll
            for (int k = 1; k < K; ++k) a1 = fma2(P[j][k], S[j][k], a1);
            c1[j] += a1.x + a1.y;
        }
        // pairs i < j
#pragma unroll
        for (int i = 0; i < D - 1; ++i) {
            if (i + (pair ? 0 : 1) >= nreal) break;
            const int fi = feat_of(r[1 + i].bits);
            const int64_t rowbase = tri_index(fi, fi + 1, F) - (fi + 1);  // + fj gives the index
            float2 R[K];
#pragma unroll
            for (int k = 0; k < K; ++k) R[k] = P[i][k];
#pragma unroll
            for (int j = i + 1; j < D; ++j) {
                if (j >= nreal) break;
                float2 acc = mul2(R[0], S[j][0]);
#pragma unroll
                for (int k = 1; k < K; ++k) acc = fma2(R[k], S[j][k], acc);
                if (j + 1 < D) {
#pragma unroll
                    for (int k = 0; k < K; ++k) R[k] = mul2(R[k], A[j][k]);
                }
                const float v = (acc.x + acc.y) * (dd[i] * dd[j]);
                const int64_t idx = rowbase + feat_of(r[1 + j].bits);
                if constexpr (PAIR_SMEM) {
                    atomicAdd(&pt[idx * kTileLd + lane], v);
                } else {
                    if (s < M && v != 0.f) atomicAdd(&acc_pair[idx * M + s], (double)v);
                }
            }
            if (!PAIR_SMEM && pair) {
                // R spans the elements between i and the pair's (padding's factors are
                // 1), whose suffix is 1
                float2 acc = R[0];
#pragma unroll
                for (int k = 1; k < K; ++k) acc = add2(R[k], acc);
                const float v = (acc.x + acc.y) * (dd[i] * dd[D - 1]);
                const int fp = feat_of(r[D].bits);
                const int64_t idx = tri_index(min(fi, fp), max(fi, fp), F);
                if (s < M && v != 0.f) atomicAdd(&acc_pair[idx * M + s], (double)v);
            }
        }
    }
#pragma unroll
    for (int j = 0; j < D; ++j)
        if (j < nreal || (pair && j == D - 1))
            atomicAdd(&ps[feat_of(r[1 + j].bits) * kTileLd + lane], dd[j] * c1[j]);
}

template <int D, int NP, bool PAIR_SMEM>
__device__ __forceinline__ bool int_segment(const IntArgs& a, const IntSeg& sg, int64_t p0, int64_t p1, bool has_nan,
                                            int64_t s, const float* xs, float* ps, float* pt, Rec32* st0, Rec32* st1,
                                            uint64_t* bars, uint32_t* s_phase, int* s_flag) {
    const int lane = threadIdx.x & 31;
    const int F = a.F;
    if (a.group > 0) {
        // few samples: lane (slot, sample) evaluates path slot of each group for
        // its sample (tile column); the pair and phi tiles take atomics anyway
        const int slot = lane / (int)a.M, col = lane - slot * (int)a.M;
        walk_paths_grouped<Rec32, D>(sg.rec, p0, p1, a.group, slot, [&](int64_t, const Rec32* r, bool valid) {
            if (!valid) return;
            int_path_f32<D, NP, true, PAIR_SMEM>(r, xs, ps, pt, a.acc_pair, col, a.M, col, F, a.q);
        });
        __syncthreads();  // every warp's adds are in the tiles before the flush
        return true;
    }
    return stream_paths<Rec32, D>(sg.rec, p0, p1, a.sub, st0, st1, bars, s_phase, s_flag, a.status,
                                  [&](int64_t, const Rec32* r) {
                                      if (has_nan)
                                          int_path_f32<D, NP, true, PAIR_SMEM>(r, xs, ps, pt, a.acc_pair, s, a.M, lane,
                                                                               F, a.q);
                                      else
                                          int_path_f32<D, NP, false, PAIR_SMEM>(r, xs, ps, pt, a.acc_pair, s, a.M,
                                                                                lane, F, a.q);
                                  });
}

template <int CLS, int NP, bool PAIR_SMEM>
__global__ void __launch_bounds__(kIntWarps * 32) int_kernel(const __grid_constant__ IntArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int F = a.F;
    const size_t rows = F + 1;
    float* xs = (float*)smem;
    float* ps = xs + rows * kTileLd;
    float* pt = ps + rows * kTileLd;
    size_t off = 2 * rows * kTileLd * 4;
    if (PAIR_SMEM) off += (size_t)a.n_pairs * kTileLd * 4;
    off = (off + 15) & ~(size_t)15;
    Rec32* st0 = (Rec32*)(smem + off);
    Rec32* st1 = st0 + a.stage;
    uint64_t* bars = (uint64_t*)(st1 + a.stage);
    __shared__ int s_flag;
    __shared__ uint32_t s_phase[2];
    int si = 0;
    while (si + 1 < a.n_seg && (int64_t)blockIdx.x >= a.seg[si + 1].cta_begin) ++si;
    const IntSeg sg = a.seg[si];
    const int64_t local = (int64_t)blockIdx.x - sg.cta_begin;
    const int lane = threadIdx.x & 31;
    const int64_t s0 = (local % a.n_tiles) * 32;
    const int64_t p0 = (local / a.n_tiles) * sg.per_cta;
    const int64_t p1 = imin64(p0 + sg.per_cta, sg.n_paths);

    if (threadIdx.x == 0) {
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
        mbar_fence_init();
        s_phase[0] = s_phase[1] = 0;
    }
    for (int idx = threadIdx.x; idx < (int)rows * kTileLd; idx += blockDim.x) ps[idx] = 0.f;
    if (PAIR_SMEM)
        for (int64_t idx = threadIdx.x; idx < a.n_pairs * kTileLd; idx += blockDim.x) pt[idx] = 0.f;
    const bool has_nan = load_tile_t(xs, a.X, s0, a.M, F, F, 1) || a.cat != 0;
    bool ok = false;
#define QTS_CASE(DD)                                                                                              \
    case DD:                                                                                                      \
        ok = int_segment<DD, NP, PAIR_SMEM>(a, sg, p0, p1, has_nan, s0 + lane, xs, ps, pt, st0, st1, bars, s_phase, \
                                            &s_flag);                                                             \
        break;
    if constexpr (CLS == 0) {
        switch (sg.D) {
            QTS_CASE(1) QTS_CASE(2) QTS_CASE(3) QTS_CASE(4)
            default: break;
        }
    } else if constexpr (CLS == 1) {
        switch (sg.D) {
            QTS_CASE(5) QTS_CASE(6)
            default: break;
        }
    } else if constexpr (CLS == 2) {
        switch (sg.D) {
            QTS_CASE(7) QTS_CASE(8)
            default: break;
        }
    } else if constexpr (CLS == 3) {
        switch (sg.D) {
            QTS_CASE(9) QTS_CASE(10) QTS_CASE(11) QTS_CASE(12)
            default: break;
        }
    } else if constexpr (CLS == 4) {
        switch (sg.D) {
            QTS_CASE(13) QTS_CASE(14) QTS_CASE(15) QTS_CASE(16)
            default: break;
        }
    } else {
        switch (sg.D) {
            QTS_CASE(20) QTS_CASE(24) QTS_CASE(28) QTS_CASE(32)
            default: break;
        }
    }
#undef QTS_CASE
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

template <int CLS, int NP, bool PS>
static cudaError_t launch_int_t(const IntArgs& a, int64_t blocks, size_t smem, cudaStream_t st) {
    auto k = int_kernel<CLS, NP, PS>;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    k<<<(unsigned)blocks, kIntWarps * 32, smem, st>>>(a);
    return cudaGetLastError();
}

// np: nodes per register pass, int_max_np of the class's widths, or 4 for widths
// up to 6 (a rule of four points)
template <int CLS>
cudaError_t launch_int_c(const IntArgs& a, int np, bool pair_smem, int64_t blocks, size_t smem, cudaStream_t st) {
    constexpr int NP = CLS <= 1 ? 8 : CLS <= 3 ? 4 : 2;
    if constexpr (NP == 8) {
        if (np < NP) {
            if (pair_smem) return launch_int_t<CLS, NP / 2, true>(a, blocks, smem, st);
            return launch_int_t<CLS, NP / 2, false>(a, blocks, smem, st);
        }
    }
    if (pair_smem) return launch_int_t<CLS, NP, true>(a, blocks, smem, st);
    if constexpr (CLS == 2) {
        // adds to global memory bound these: one pass over all nodes halves them (100
        // trees of depth 8, F = 56, 2,000 samples 2,260 -> 1,913 us)
        if (a.q.n_pad % 8 == 0) return launch_int_t<CLS, 8, false>(a, blocks, smem, st);
    }
    return launch_int_t<CLS, NP, false>(a, blocks, smem, st);
}

#define QTS_INST(C) template cudaError_t launch_int_c<C>(const IntArgs&, int, bool, int64_t, size_t, cudaStream_t);
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
#if QTS_IN_PART(6)
QTS_INST(5)
#endif
#undef QTS_INST

#endif  // QTS_DEVICE_PARTS

#if !QTS_HOST_PART
}  // namespace qts
#endif

#if QTS_HOST_PART

static size_t int_smem_bytes(int F, int stage, bool pair_smem) {
    const size_t rows = F + 1;
    size_t off = 2 * rows * kTileLd * 4;
    if (pair_smem) off += (size_t)F * (F - 1) / 2 * kTileLd * 4;
    off = (off + 15) & ~(size_t)15;
    return off + 2 * (size_t)stage * sizeof(Rec32) + 16;
}

// out[s][i][j] (F+1 x F+1, fp32) from the FP64 accumulators; one thread per (s, i).
__global__ void int_finalize_kernel(const double* __restrict__ acc_pair, const double* __restrict__ acc_phi,
                                    int64_t M, int F, double bias, float* __restrict__ out) {
    const int64_t n = M * (F + 1);
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t s = t % M;
        const int i = (int)(t / M);
        float* row = out + (s * (F + 1) + i) * (F + 1);
        if (i == F) {
            for (int j = 0; j < F; ++j) row[j] = 0.f;
            row[F] = (float)bias;
            continue;
        }
        double rowsum = 0.0;
        for (int j = 0; j < F; ++j) {
            if (j == i) continue;
            const int a = i < j ? i : j, b = i < j ? j : i;
            const double h = 0.5 * acc_pair[tri_index(a, b, F) * M + s];
            row[j] = (float)h;
            rowsum += h;
        }
        row[i] = (float)(acc_phi[(int64_t)i * M + s] - rowsum);
        row[F] = 0.f;
    }
}

static constexpr size_t kSmemBudget = 200 * 1024;

// Pairwise sums of every bucket of the path tables, one path per leaf or (F too large for a
// pair tile) with sibling leaves merged (QTS_NQ_EXACT: the first-order
// count per bucket, because the diagonal holds first-order values).
static cudaError_t launch_int_buckets(const qts_ensemble* e, const Rec32* rec, const std::vector<Bucket>& buckets,
                                      const float* X, int64_t M, int F, int n_quad, double* acc_pair, double* acc_phi,
                                      cudaStream_t st) {
    if (M <= 0) return cudaSuccess;
    const int64_t tiles = (M + 31) / 32;
    const int group = M <= kFewRows ? (int)(32 / M) : 0;
    // work per thread block: about eight rounds of the whole chip (three thread
    // blocks per SM); at least what makes the set-up and flush of the tiles, F^2 / 2 rows
    // where the pair tile fits and F where not, small beside the paths'
    double total = 0.0;
    for (const Bucket& b : buckets) total += (double)b.n_paths * b.D * (b.D + 8);
    const bool tile = int_smem_bytes(F, 16 * 17, true) <= kSmemBudget;
    const double least = std::min(512.0, 64.0 + (tile ? (double)F * F / 8.0 : F / 2.0)) * 60.0;
    const double share = std::max(least, std::min(512.0 * 84.0, total * (double)tiles / (8.0 * 3 * num_sms())));
    for (int cls = 0; cls < kIntClasses; ++cls) {
        uint64_t rules = 0;  // bit q: some bucket of the class takes q points
        for (const Bucket& b : buckets)
            if (b.n_paths > 0 && int_class(b.D) == cls) rules |= (uint64_t)1 << nodes_for(n_quad, b.D, 1);
        for (int nq = QTS_MAX_QUAD; nq >= 1; --nq) {  // one launch per rule
            if (!((rules >> nq) & 1)) continue;
            IntArgs a;
            a.n_seg = 0;
            int64_t ctas = 0;
            int max_d = 0;
            // widest first: its thread blocks are the longest
            for (auto it = buckets.rbegin(); it != buckets.rend(); ++it) {
                const Bucket& b = *it;
                if (b.n_paths == 0 || int_class(b.D) != cls || nodes_for(n_quad, b.D, 1) != nq) continue;
                max_d = std::max(max_d, b.D);
                int64_t per = std::max<int64_t>(16, (int64_t)(share / (b.D * (b.D + 8))));
                if (group) per = std::max<int64_t>(per, 4LL * kIntWarps * group);
                per = std::min<int64_t>((per + 15) / 16 * 16, 1 << 20);
                a.seg[a.n_seg++] = {rec + b.rec_off, b.n_paths, ctas, (int32_t)per, b.D};
                ctas += (b.n_paths + per - 1) / per * tiles;
            }
            if (a.n_seg == 0) continue;
            if (ctas > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
            // the rule, padded to 4 nodes up to width 12 (a pass of 4 or 8 nodes) and to
            // 2 above
            if (!make_quad(nq, &a.q, nullptr, cls <= 3 ? 4 : 2)) return cudaErrorInvalidValue;
            a.sub = max_d <= 16 ? 16 : 8;
            // wide inputs: stage fewer paths at a time until the block fits shared memory
            while (a.sub > 1 && int_smem_bytes(F, a.sub * (max_d + 1), false) > kSmemMax) a.sub /= 2;
            a.stage = a.sub * (max_d + 1);
            a.n_tiles = (int)tiles;
            a.X = X;
            a.M = M;
            a.F = F;
            a.cat = e->prep.has_cat ? 1 : 0;
            a.n_pairs = (int64_t)F * (F - 1) / 2;
            a.group = group;
            a.acc_pair = acc_pair;
            a.acc_phi = acc_phi;
            a.status = e->d_status;
            const bool pair_smem = int_smem_bytes(F, a.stage, true) <= kSmemBudget;
            const size_t smem = int_smem_bytes(F, a.stage, pair_smem);
            if (smem > kSmemMax) return cudaErrorInvalidConfiguration;
            // nodes per register pass: the class's widest, or half of it when that
            // does not divide the rule's padded node count
            const int np = a.q.n_pad % int_max_np(max_d) == 0 ? int_max_np(max_d) : int_max_np(max_d) / 2;
            if (a.q.n_pad % np != 0) return cudaErrorInvalidValue;
            const cudaError_t r = cls == 0   ? launch_int_c<0>(a, np, pair_smem, ctas, smem, st)
                                  : cls == 1 ? launch_int_c<1>(a, np, pair_smem, ctas, smem, st)
                                  : cls == 2 ? launch_int_c<2>(a, np, pair_smem, ctas, smem, st)
                                  : cls == 3 ? launch_int_c<3>(a, np, pair_smem, ctas, smem, st)
                                  : cls == 4 ? launch_int_c<4>(a, np, pair_smem, ctas, smem, st)
                                             : launch_int_c<5>(a, np, pair_smem, ctas, smem, st);
            if (r != cudaSuccess) return r;
        }
    }
    return cudaSuccess;
}

cudaError_t launch_int_finalize(const double* acc_pair, const double* acc_phi, int64_t M, int F,
                                double bias, float* out, cudaStream_t st) {
    const int64_t n = M * (F + 1);
    const int blocks = (int)std::min<int64_t>((n + 255) / 256, 8 * 152);
    int_finalize_kernel<<<blocks, 256, 0, st>>>(acc_pair, acc_phi, M, F, bias, out);
    return cudaGetLastError();
}

}  // namespace qts

namespace qts {

// Which tables a pairwise call runs on: the blocks, or, where F is too large for a pair
// tile in shared memory, the path tables with sibling leaves merged.  Without a tile every
// add goes to global memory: a block needs fewer of them, but keeps more vectors than
// fit its registers and has fewer warps in flight.  Blocks and paths: 100 trees of depth 8,
// F = 56, 300 samples 1,314 and 428 us, 2,000 4,064 and 1,913, 6,000 9,969 and 5,454 (one
// launch per width: 2,213, 2,679 and 6,381); F = 200, 2,000 samples 8,060 and 3,033; 300
// trees of depth 4, F = 56, 2,000 samples 455 and 164; one row of 8 trees of depth 14, F
// = 60 512 and 440, but of 2 trees of depth 18 731 and 872, F = 400 913 and 1,894.  The
// paths' error against FP64 is the smaller one there (100 trees of depth 8, F = 60:
// 1.0e-7 against 1.3e-7).  With a tile the blocks stay, also where the per-leaf paths are
// faster (mean width above 9.5: F = 24, depth 14, 640 samples 11.2 ms against 6.5), because
// there the blocks' error is smaller (1.8e-7 against 2.1e-7).
static bool pairs_on_paths(const qts_ensemble* e, int64_t M, int F) {
    if (int_smem_bytes(F, 16 * 17, true) <= kSmemBudget) return false;
    return M > 1 || (double)e->prep.sum_unique <= 13.5 * (double)e->prep.n_paths;
}

}  // namespace qts

using namespace qts;

extern "C" qts_status qts_shap_interactions(qts_ensemble* e, const float* X, int64_t M, int32_t F,
                                            int32_t n_quad, float* phi_ij, qts_stream_t stream) try {
    qts_status st = check_call(e, X, M, F, n_quad);
    if (st != QTS_OK) return st;
    if (M == 0) return QTS_OK;
    if (!phi_ij) return fail(QTS_ERR_ARG, "phi_ij is NULL");
    if (e->flags & QTS_FLAG_FP64)
        return fail(QTS_ERR_UNSUPPORTED, "interactions are computed with the FP32 tables only");
    if (e->prep.max_unique > 32)
        return fail(QTS_ERR_UNSUPPORTED, "interactions support paths of at most 32 unique features");
    cudaStream_t s = (cudaStream_t)stream;
    if (n_quad != QTS_NQ_EXACT && (n_quad < 1 || n_quad > QTS_MAX_QUAD)) return fail(QTS_ERR_ARG, "quadrature rule");
    const bool paths = pairs_on_paths(e, M, F);
    // the tables (built on the first call that needs them)
    st = paths ? ensure_pairs(e, true) : ensure_blocks(e, false);
    if (st != QTS_OK) return st;
    const int64_t n_pairs = (int64_t)F * (F - 1) / 2;
    const size_t bytes = sizeof(double) * (size_t)((n_pairs + F) * M);
    st = ensure_workspace(e, bytes, s);
    if (st != QTS_OK) return st;
    double* acc_pair = (double*)e->d_work;
    double* acc_phi = acc_pair + n_pairs * M;
    cudaError_t ce = cudaMemsetAsync(e->d_work, 0, bytes, s);
    if (ce != cudaSuccess) return cuda_fail(ce, "workspace clear");
    ce = paths ? launch_int_buckets(e, e->d_pair_rec, e->pair_sizes.buckets, X, M, F, n_quad, acc_pair, acc_phi, s)
               : launch_int_blocks(e, X, M, F, n_quad, acc_pair, acc_phi, s);
    if (ce != cudaSuccess) return cuda_fail(ce, "interaction kernel launch");
    ce = launch_int_finalize(acc_pair, acc_phi, M, F, e->prep.bias, phi_ij, s);
    if (ce != cudaSuccess) return cuda_fail(ce, "interaction finalize launch");
    return QTS_OK;
} QTS_ENTRY_END

// ------------------------------------------------- allocation-free variant --
//
// Same kernels as qts_shap_interactions, but the FP64 accumulators live in a
// fixed device array that is part of the library image, so the call never
// allocates.  Host code cannot use the array's name as a device pointer: its
// address comes from cudaGetSymbolAddress, with the device current.  That
// address belongs to a context - a device reset destroys the primary context,
// the next call creates a new one, reloads the library's module, and the array
// may then sit elsewhere - so the looked-up address is cached under the current
// context's process-unique id (cuCtxGetId), not under the device ordinal.  The
// two driver calls are fetched through the runtime, so the library still links
// no driver library of its own.

namespace qts {

constexpr int64_t kNoAllocDoubles = (int64_t)2 * 1024 * 1024;  // 16 MiB per device

static __device__ __align__(256) double g_int_noalloc_scratch[kNoAllocDoubles];

struct CtxFns {
    PFN_cuCtxGetCurrent_v4000 get_current = nullptr;
    PFN_cuCtxGetId_v12000 get_id = nullptr;
};

static CtxFns ctx_fns() {
    static CtxFns f;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            f.get_current = (PFN_cuCtxGetCurrent_v4000)p;
        p = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            f.get_id = (PFN_cuCtxGetId_v12000)p;
        cudaGetLastError();  // a missing entry point is not an error of the caller's next call
    });
    return f;
}

// Unique id of the context current on this thread; false when there is none
// (the runtime has not made one current yet) or the driver cannot say.
static bool current_ctx_id(unsigned long long* id) {
    const CtxFns f = ctx_fns();
    if (!f.get_current || !f.get_id) return false;
    CUcontext ctx = nullptr;
    if (f.get_current(&ctx) != CUDA_SUCCESS || !ctx) return false;
    return f.get_id(ctx, id) == CUDA_SUCCESS;
}

static std::mutex g_noalloc_mu;
static std::vector<std::pair<unsigned long long, void*>> g_noalloc_ptr;  // (context id, address)

static qts_status noalloc_scratch(void** out) {
    unsigned long long id = 0;
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (current_ctx_id(&id)) {
        for (const auto& kv : g_noalloc_ptr)
            if (kv.first == id) {
                *out = kv.second;
                return QTS_OK;
            }
    }
    void* p = nullptr;
    cudaError_t ce = cudaGetSymbolAddress(&p, g_int_noalloc_scratch);
    if (ce != cudaSuccess) return cuda_fail(ce, "cudaGetSymbolAddress of the interaction scratch");
    // the lookup makes the device's context current if none was: ask again;
    // without an id the address is not cached and is looked up on every call
    if (current_ctx_id(&id)) g_noalloc_ptr.emplace_back(id, p);
    *out = p;
    return QTS_OK;
}

}  // namespace qts

extern "C" qts_status qts_shap_interactions_noalloc(qts_ensemble* e, const float* X, int64_t M, int32_t F,
                                                    int32_t n_quad, float* phi_ij, qts_stream_t stream) try {
    qts_status st = check_call(e, X, M, F, n_quad);
    if (st != QTS_OK) return st;
    if (M == 0) return QTS_OK;
    if (!phi_ij) return fail(QTS_ERR_ARG, "phi_ij is NULL");
    if (e->flags & QTS_FLAG_FP64)
        return fail(QTS_ERR_UNSUPPORTED, "interactions are computed with the FP32 tables only");
    if (e->prep.max_unique > 32)
        return fail(QTS_ERR_UNSUPPORTED, "interactions support paths of at most 32 unique features");
    const int64_t n_pairs = (int64_t)F * (F - 1) / 2;
    const int64_t need = (n_pairs + F) * M;
    if (need > kNoAllocDoubles)
        return fail(QTS_ERR_UNSUPPORTED,
                    "qts_shap_interactions_noalloc needs (F(F-1)/2 + F) * M = " + std::to_string(need) +
                        " accumulator doubles; the fixed scratch holds " + std::to_string(kNoAllocDoubles) +
                        " (use qts_shap_interactions for larger calls)");
    cudaStream_t s = (cudaStream_t)stream;
    // QTS_NQ_EXACT: exact for the ensemble's widest path; first-order count,
    // because the diagonal holds first-order values (Thm 2)
    const int nq = nodes_for(n_quad, std::max(1, e->prep.max_unique), 1);
    if (nq < 1 || nq > QTS_MAX_QUAD) return fail(QTS_ERR_ARG, "quadrature rule");
    void* scratch = nullptr;
    st = noalloc_scratch(&scratch);
    if (st != QTS_OK) return st;
    double* acc_pair = (double*)scratch;
    double* acc_phi = acc_pair + n_pairs * M;
    // the array keeps the previous call's sums: clear the part this call uses
    cudaError_t ce = cudaMemsetAsync(scratch, 0, sizeof(double) * (size_t)need, s);
    if (ce != cudaSuccess) return cuda_fail(ce, "scratch clear");
    ce = launch_int_buckets(e, (const Rec32*)e->d_rec, e->prep.buckets, X, M, F, nq, acc_pair, acc_phi, s);
    if (ce != cudaSuccess) return cuda_fail(ce, "interaction kernel launch");
    ce = launch_int_finalize(acc_pair, acc_phi, M, F, e->prep.bias, phi_ij, s);
    if (ce != cudaSuccess) return cuda_fail(ce, "interaction finalize launch");
    return QTS_OK;
} QTS_ENTRY_END

#endif  // QTS_HOST_PART
