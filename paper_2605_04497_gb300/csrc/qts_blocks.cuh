// Device evaluation of blocks (layout and formulation: qts_blocks.h).
#pragma once

#include "qts_blocks.h"
#include "qts_paths.cuh"

namespace qts {

// one record as four floats
__device__ __forceinline__ float4 rec4(const Rec32* r) { return *reinterpret_cast<const float4*>(r); }

// Whether a sample takes a node's left edge, its right edge.  Only a block's root
// (ROOT) can have an interval left by splits above it.
template <bool ROOT, bool HAS_NAN>
__device__ __forceinline__ void node_sides(float x, const float4& b, bool* l, bool* r) {
    const uint32_t bits = __float_as_uint(b.w);
    bool in = !ROOT || (x >= b.y && x < b.z), left = x < b.x;
    if (HAS_NAN && x != x) {
        in = !ROOT || (bits & kNanOk) != 0;
        left = (bits & kDefLeft) != 0;
    }
    *l = in && left;
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

}  // namespace qts
