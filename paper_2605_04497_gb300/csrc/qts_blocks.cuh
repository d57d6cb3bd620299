// Device evaluation of blocks (layout and formulation: qts_blocks.h).
#pragma once

#include "qts_blocks.h"
#include "qts_paths.cuh"

namespace qts {

// one record as four floats
__device__ __forceinline__ float4 rec4(const Rec32* r) { return *reinterpret_cast<const float4*>(r); }

// Whether a sample takes a node's left edge, its right edge.  Only a block's root
// (ROOT) can have an interval left by splits above it; below it hi = +inf still
// excludes x = +inf, as the path tables' half-open intervals do (HAS_NAN: some
// value of the tile is NaN or +inf, so the others need no test).
template <bool ROOT, bool HAS_NAN>
__device__ __forceinline__ void node_sides(float x, const float4& b, bool* l, bool* r) {
    bool in = true, left = x < b.x;
    if (ROOT) in = x >= b.y && x < b.z;
    else if (HAS_NAN) in = x < b.z;
    if (HAS_NAN && x != x) {
        const uint32_t bits = __float_as_uint(b.w);
        in = !ROOT || (bits & kNanOk) != 0;
        left = (bits & kDefLeft) != 0;
    }
    *l = ROOT ? in && left : left;  // below the root, theta <= hi: left implies x < hi
    *r = in && !left;
}

// ====================================================== first order ======
//
// Lane = sample, NP = 2 K quadrature nodes per pass, two to an f32x2 register
// pair.

template <int K>
__device__ __forceinline__ float dot_k(const float2 (&u)[K], const float2 (&v)[K]) {
    float2 s = mul2(u[0], v[0]);
#pragma unroll
    for (int k = 1; k < K; ++k) s = fma2(u[k], v[k], s);
    return s.x + s.y;
}

// G = the sum over node N's leaves of val times the factors met from N down, at
// the pass's quadrature nodes T; C = the product of the factors above (and the
// weights).  Adds the subtree's contributions to phi.
template <int H, int N, int LEVELS, int K, bool HAS_NAN, int PHI, typename XR>
__device__ __forceinline__ void fwd_node(const Rec32* nodes, const XR& xr, float* ps, int lane, const float2 (&T)[K],
                                         const float2 (&C)[K], float2 (&G)[K]) {
    const float4 a = rec4(nodes + blk_rec(H, N)), b = rec4(nodes + blk_rec(H, N) + 1);
    const int f = feat_of(__float_as_uint(b.w));
    bool l, r;
    node_sides<N == 1, HAS_NAN>(xr(f), b, &l, &r);
    if constexpr (LEVELS == 1) {
        const float vd = fmaf(a.x, (l ? 1.f : 0.f) - a.z, a.y * ((r ? 1.f : 0.f) - a.w));
        const float vz = nodes[blk_rec(H, N) + 2].z;
        float2 s = C[0];
#pragma unroll
        for (int k = 1; k < K; ++k) s = add2(s, C[k]);
#pragma unroll
        for (int k = 0; k < K; ++k) G[k] = fma2(T[k], f2s(vd), f2s(vz));
        phi_add<PHI>(ps, f * kTileLd + lane, vd * (s.x + s.y));
    } else {
        const float dL = (l ? 1.f : 0.f) - a.x, dR = (r ? 1.f : 0.f) - a.z;
        float2 A[K], Q[K], GC[K];
        auto side = [&](auto child, float d, float z, bool first) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                A[k] = fma2(T[k], f2s(d), f2s(z));
                Q[k] = mul2(C[k], A[k]);
            }
            fwd_node<H, decltype(child)::value, LEVELS - 1, K, HAS_NAN, PHI>(nodes, xr, ps, lane, T, Q, GC);
#pragma unroll
            for (int k = 0; k < K; ++k) G[k] = first ? mul2(A[k], GC[k]) : fma2(A[k], GC[k], G[k]);
            return d * dot_k<K>(C, GC);
        };
        float ph = side(std::integral_constant<int, 2 * N>{}, dL, a.x, true);
        ph += side(std::integral_constant<int, 2 * N + 1>{}, dR, a.z, false);
        phi_add<PHI>(ps, f * kTileLd + lane, ph);
    }
}

// One block of width D and height H: the shared elements by a prefix product
// seeded with w_m and a suffix product that starts at the subtree's sum.
template <int D, int H, int NP, bool HAS_NAN, int PHI, typename XR>
__device__ __forceinline__ void fwd_block(const Rec32* __restrict__ r, const XR& xr, float* ps, int lane,
                                          const QuadF& q) {
    constexpr int K = NP / 2;
    constexpr int DN = D > 0 ? D : 1;
    const uint32_t* words = reinterpret_cast<const uint32_t*>(r + 1 + D);
    float dd[DN], zz[DN], cacc[DN];
#pragma unroll
    for (int j = 0; j < D; ++j) {
        const float4 e = rec4(r + 1 + j);
        const uint32_t word = words[j];
        dd[j] = (satisfies<HAS_NAN>(xr(feat_of(word)), e.z, e.w, word) ? 1.f : 0.f) - e.x;
        zz[j] = e.x;
        cacc[j] = 0.f;
    }
    for (int m0 = 0; m0 < q.n_pad; m0 += NP) {
        float2 T[K], P[D + 1][K], G[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            T[k] = f2(q.t[m0 + 2 * k], q.t[m0 + 2 * k + 1]);
            P[0][k] = f2(q.w[m0 + 2 * k], q.w[m0 + 2 * k + 1]);
        }
#pragma unroll
        for (int j = 0; j < D; ++j)
#pragma unroll
            for (int k = 0; k < K; ++k) P[j + 1][k] = mul2(P[j][k], fma2(T[k], f2s(dd[j]), f2s(zz[j])));
        if constexpr (H > 0) {
            fwd_node<H, 1, H, K, HAS_NAN, PHI>(r + blk_head(D), xr, ps, lane, T, P[D], G);
        } else {
#pragma unroll
            for (int k = 0; k < K; ++k) G[k] = f2s(r[0].z);
        }
#pragma unroll
        for (int j = D - 1; j >= 0; --j) {
            cacc[j] += dot_k<K>(P[j], G);
            if (j > 0) {
#pragma unroll
                for (int k = 0; k < K; ++k) G[k] = mul2(G[k], fma2(T[k], f2s(dd[j]), f2s(zz[j])));
            }
        }
    }
#pragma unroll
    for (int j = 0; j < D; ++j) phi_add<PHI>(ps, feat_of(words[j]) * kTileLd + lane, dd[j] * cacc[j]);
}

// ============================================= first order and adjoint ==
//
// Forward values and the adjoint in one sweep (formulation: qts_bwd.cu) with dual
// numbers: C carries CU = sum over the elements i in it of u_i prod_{l != i} a_l,
// and G carries GU likewise.  For an edge with factor a and leaf sum G below it
//     dL/da = sum_m w_m (C GU + CU G),  dL/du = sum_m w_m C G = its phi / d.
// Every f32x2 operation covers two samples at one node (SP: lane l holds samples
// 2l, 2l + 1 of 64, so record loads, addresses and the warp reduction serve 64
// samples) or two nodes of one sample (requests whose 64-sample tile would not
// fit).  All state lies in registers under compile-time indices.

template <bool SP>
struct BwdCols {  // one sample's (or pair's) column of a transposed global copy
    const float* t;
    int64_t ld;
    int64_t s;
    __device__ __forceinline__ float2 operator()(int f) const {
        const float* p = t + (int64_t)f * ld + s;
        if constexpr (SP) return __ldg(reinterpret_cast<const float2*>(p));
        else return f2s(__ldg(p));
    }
};

template <bool SP, int PHI>
__device__ __forceinline__ void phi_add2(float* ps, int f, int lane, float2 v) {
    if constexpr (SP) {
        float2* cell = reinterpret_cast<float2*>(ps + f * kTileLd2 + 2 * lane);
        *cell = add2(*cell, v);  // this warp's own tile
    } else {
        phi_add<PHI>(ps, f * kTileLd + lane, v.x + v.y);
    }
}

// {z, z} as the records hold it, re-read at every use (see lds_pair)
__device__ __forceinline__ float2 zpair(const Rec32* r, int half) {
    return lds_pair(reinterpret_cast<const float2*>(r) + half);
}

template <int H, bool HAS_NAN, bool SP>
struct BwdTree {
    struct Inner { float2 dL, dR, uL, uR, a1L, a2L, a1R, a2R; };
    struct Pair { float2 vd, gv, q1, q2, q3; };
    const Rec32* nodes;
    Inner in[blk_inner(H) > 0 ? blk_inner(H) : 1];
    Pair pr[blk_pairs(H) > 0 ? blk_pairs(H) : 1];

    template <int N>
    __device__ __forceinline__ void sides(const BwdCols<SP>& xr, int* f, float2* l, float2* r) const {
        const float4 b = rec4(nodes + blk_rec(H, N) + 1);
        *f = feat_of(__float_as_uint(b.w));
        const float2 x = xr(*f);
        bool l0, r0, l1, r1;
        node_sides<N == 1, HAS_NAN>(x.x, b, &l0, &r0);
        node_sides<N == 1, HAS_NAN>(x.y, b, &l1, &r1);
        *l = f2(l0 ? 1.f : 0.f, l1 ? 1.f : 0.f);
        *r = f2(r0 ? 1.f : 0.f, r1 ? 1.f : 0.f);
    }

    template <int N, int LEVELS>
    __device__ __forceinline__ void decode(const BwdCols<SP>& xr, const BwdCols<SP>& gr) {
        const float4 a = rec4(nodes + blk_rec(H, N));
        int f;
        float2 l, r;
        sides<N>(xr, &f, &l, &r);
        const float2 g = gr(f);
        if constexpr (LEVELS == 1) {
            Pair& s = pr[N - 1 - blk_inner(H)];
            s.vd = fma2(f2s(a.x), add2(l, f2s(-a.z)), mul2(f2s(a.y), add2(r, f2s(-a.w))));
            s.gv = mul2(g, s.vd);
            s.q1 = s.q2 = s.q3 = f2s(0.f);
        } else {
            Inner& s = in[N - 1];
            s.dL = add2(l, f2s(-a.x));
            s.dR = add2(r, f2s(-a.z));
            s.uL = mul2(g, s.dL);
            s.uR = mul2(g, s.dR);
            s.a1L = s.a2L = s.a1R = s.a2R = f2s(0.f);
            decode<2 * N, LEVELS - 1>(xr, gr);
            decode<2 * N + 1, LEVELS - 1>(xr, gr);
        }
    }

    template <int N, int LEVELS>
    __device__ __forceinline__ void eval(float2 T, float2 T1, float2 C, float2 CU, float2& G, float2& GU) {
        if constexpr (LEVELS == 1) {
            Pair& s = pr[N - 1 - blk_inner(H)];
            G = fma2(T, s.vd, zpair(nodes + blk_rec(H, N) + 2, 0));
            GU = s.gv;
            s.q1 = add2(s.q1, C);
            s.q2 = add2(s.q2, CU);
            s.q3 = fma2(T1, CU, s.q3);
        } else {
            Inner& s = in[N - 1];
            float2 g, gu;
            {
                const float2 a = fma2(T, s.dL, zpair(nodes + blk_rec(H, N), 0));
                eval<2 * N, LEVELS - 1>(T, T1, mul2(C, a), fma2(CU, a, mul2(s.uL, C)), g, gu);
                s.a1L = fma2(C, g, s.a1L);
                s.a2L = fma2(T1, fma2(C, gu, mul2(CU, g)), s.a2L);
                G = mul2(a, g);
                GU = fma2(a, gu, mul2(s.uL, g));
            }
            {
                const float2 a = fma2(T, s.dR, zpair(nodes + blk_rec(H, N), 1));
                eval<2 * N + 1, LEVELS - 1>(T, T1, mul2(C, a), fma2(CU, a, mul2(s.uR, C)), g, gu);
                s.a1R = fma2(C, g, s.a1R);
                s.a2R = fma2(T1, fma2(C, gu, mul2(CU, g)), s.a2R);
                G = fma2(a, g, G);
                GU = fma2(a, gu, fma2(s.uR, g, GU));
            }
        }
    }

    // phi of the subtree's features and this lane's share of its adjoint sums
    template <int N, int LEVELS, int PHI>
    __device__ __forceinline__ void finish(const BwdCols<SP>& xr, const BwdCols<SP>& gr, float* ps, int lane,
                                           float* v) {
        int f;
        float* o = v + blk_slot(H, N);
        if constexpr (LEVELS == 1) {
            const Pair& s = pr[N - 1 - blk_inner(H)];
            float2 l, r;
            sides<N>(xr, &f, &l, &r);
            const float2 q = fma2(f2s(-1.f), mul2(gr(f), s.q1), s.q3);
            const float2 k = fma2(f2s(-1.f), q, s.q2);
            const float2 kl = mul2(l, k), kr = mul2(r, k);
            o[0] = q.x + q.y;
            o[1] = kl.x + kl.y;
            o[2] = kr.x + kr.y;
            phi_add2<SP, PHI>(ps, f, lane, mul2(s.vd, s.q1));
        } else {
            const Inner& s = in[N - 1];
            f = feat_of(nodes[blk_rec(H, N) + 1].bits);
            const float2 g = gr(f);
            const float2 zl = fma2(f2s(-1.f), mul2(g, s.a1L), s.a2L), zr = fma2(f2s(-1.f), mul2(g, s.a1R), s.a2R);
            o[0] = zl.x + zl.y;
            o[1] = zr.x + zr.y;
            phi_add2<SP, PHI>(ps, f, lane, fma2(s.dL, s.a1L, mul2(s.dR, s.a1R)));
            finish<2 * N, LEVELS - 1, PHI>(xr, gr, ps, lane, v);
            finish<2 * N + 1, LEVELS - 1, PHI>(xr, gr, ps, lane, v);
        }
    }
};

// Sum v[0..N) over the warp and add it to g[0..N) (FP64).
template <int N>
__device__ __forceinline__ void flush_slots(float (&v)[N], int lane, double* g) {
    if constexpr (N <= 32) {
        constexpr int P = pow2_at_least(N);
        constexpr int LOG = (P >= 32) ? 5 : (P >= 16) ? 4 : (P >= 8) ? 3 : (P >= 4) ? 2 : (P >= 2) ? 1 : 0;
        float w[P];
#pragma unroll
        for (int i = 0; i < P; ++i) w[i] = i < N ? v[i] : 0.f;
        const float r = transpose_reduce<P>(w, lane);
        const int idx = lane >> (5 - LOG);
        if ((lane & ((1 << (5 - LOG)) - 1)) == 0 && idx < N) atomicAdd(&g[idx], (double)r);
    } else {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            float x = v[i];
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
            if (lane == 0) atomicAdd(&g[i], (double)x);
        }
    }
}

template <int D, int H, bool HAS_NAN, bool SP, int PHI>
__device__ __forceinline__ void bwd_block(const Rec32* __restrict__ r, const BwdCols<SP>& xr, const BwdCols<SP>& gr,
                                          float* ps, int lane, const QuadF& q, double* g_blk) {
    constexpr int DN = D > 0 ? D : 1;
    const uint32_t* words = reinterpret_cast<const uint32_t*>(r + 1 + D);
    float2 d[DN], u[DN], a1[DN], a2[DN], q0 = f2s(0.f);
    BwdTree<H, HAS_NAN, SP> t;
    t.nodes = r + blk_head(D);
#pragma unroll
    for (int j = 0; j < D; ++j) {
        const float4 e = rec4(r + 1 + j);
        const uint32_t word = words[j];
        const int f = feat_of(word);
        const float2 x = xr(f);
        const bool oa = satisfies<HAS_NAN>(x.x, e.z, e.w, word), ob = satisfies<HAS_NAN>(x.y, e.z, e.w, word);
        d[j] = f2((oa ? 1.f : 0.f) - e.x, (ob ? 1.f : 0.f) - e.x);
        u[j] = mul2(gr(f), d[j]);
        a1[j] = a2[j] = f2s(0.f);
    }
    if constexpr (H > 0) t.template decode<1, H>(xr, gr);
    const float val = r[0].z;
#pragma unroll 1
    for (int m = 0; m < q.n_pad; m += SP ? 1 : 2) {
        const float2 T = SP ? f2s(q.t[m]) : f2(q.t[m], q.t[m + 1]);
        const float2 T1 = SP ? f2s(1.f - q.t[m]) : f2(1.f - q.t[m], 1.f - q.t[m + 1]);
        float2 P[D + 1], PU[D + 1], S, SU;
        P[0] = SP ? f2s(q.w[m]) : f2(q.w[m], q.w[m + 1]);
        PU[0] = f2s(0.f);
#pragma unroll
        for (int j = 0; j < D; ++j) {
            const float2 a = fma2(T, d[j], zpair(r + 1 + j, 0));
            P[j + 1] = mul2(P[j], a);
            PU[j + 1] = fma2(PU[j], a, mul2(u[j], P[j]));
        }
        if constexpr (H > 0) {
            t.template eval<1, H>(T, T1, P[D], PU[D], S, SU);
        } else {
            S = f2s(val);
            SU = f2s(0.f);
            q0 = add2(q0, PU[D]);
        }
#pragma unroll
        for (int j = D - 1; j >= 0; --j) {
            a1[j] = fma2(P[j], S, a1[j]);
            a2[j] = fma2(T1, fma2(P[j], SU, mul2(PU[j], S)), a2[j]);
            if (j > 0) {
                const float2 a = fma2(T, d[j], zpair(r + 1 + j, 0));
                SU = fma2(SU, a, mul2(u[j], S));
                S = mul2(S, a);
            }
        }
    }
    float v[D + blk_slots(H)];
#pragma unroll
    for (int j = 0; j < D; ++j) {
        const int f = feat_of(words[j]);
        const float2 z = fma2(f2s(-1.f), mul2(gr(f), a1[j]), a2[j]);
        v[j] = z.x + z.y;
        phi_add2<SP, PHI>(ps, f, lane, mul2(d[j], a1[j]));
    }
    if constexpr (H > 0) t.template finish<1, H, PHI>(xr, gr, ps, lane, v + D);
    else v[D] = q0.x + q0.y;
    flush_slots<D + blk_slots(H)>(v, lane, g_blk);
}

}  // namespace qts
