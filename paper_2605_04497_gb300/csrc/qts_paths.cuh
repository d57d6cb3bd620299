// Per-path device routines shared by the per-bucket kernels and the batched
// persistent kernel.  Lane = sample; all path records are warp-uniform.
#pragma once

#include <type_traits>

#include "qts_device.cuh"

namespace qts {

// How a path adds its phi contributions to the shared tile.
// kPhiAtomicNz skips zeros: lanes that hold different blocks meet at the zero
// row of absent elements, where atomics would serialise.
enum PhiMode : int { kPhiAtomic = 1, kPhiPrivate = 2, kPhiAtomicNz = 3 };

template <int MODE>
__device__ __forceinline__ void phi_add(float* ps, int idx, float v) {
    if constexpr (MODE == kPhiAtomic) atomicAdd(&ps[idx], v);
    else if constexpr (MODE == kPhiPrivate) ps[idx] += v;  // tile owned by this warp
    else if (v != 0.f) atomicAdd(&ps[idx], v);
}

// Per-lane reads of one sample's values by feature index.
struct SmemCols {  // transposed shared tile [feature][kTileLd]; column = lane
    const float* t;
    int lane;
    __device__ __forceinline__ float operator()(int f) const { return t[f * kTileLd + lane]; }
};
struct GlobalCols {  // transposed global copy [feature][ld]; this lane's sample = s
    const float* t;
    int64_t ld;
    int64_t s;
    __device__ __forceinline__ float operator()(int f) const { return __ldg(t + (int64_t)f * ld + s); }
};

// =========================================================== adjoint =====

// ------------------------------------------------- warp transpose-reduce --
//
// Each lane holds N values (N a power of two <= 32).  log2(N) halving steps
// exchange half of the values with the partner lane at distance 16, 8, ...,
// keeping the other half, so that after them lane L holds, summed over a group
// of lanes, the value with index L >> (5 - log2 N); the remaining distances
// finish the sum.  N - 1 + (5 - log2 N) shuffles instead of 5 N.
template <int N>
__device__ __forceinline__ float transpose_reduce(float (&v)[N], int lane) {
    static_assert(N >= 1 && N <= 32 && (N & (N - 1)) == 0, "N must be a power of two <= 32");
#pragma unroll
    for (int half = N / 2, off = 16; half >= 1; half >>= 1, off >>= 1) {
        const bool upper = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const float send = upper ? v[i] : v[i + half];
            const float keep = upper ? v[i + half] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
    float r = v[0];
    constexpr int LOG = (N >= 32) ? 5 : (N >= 16) ? 4 : (N >= 8) ? 3 : (N >= 4) ? 2 : (N >= 2) ? 1 : 0;
#pragma unroll
    for (int off = (16 >> LOG); off >= 1; off >>= 1) r += __shfl_xor_sync(0xffffffffu, r, off);
    return r;
}

constexpr int pow2_at_least(int x) { return x <= 1 ? 1 : 2 * pow2_at_least((x + 1) / 2); }

// Reduce dz[0..D) and dval over the warp and add them to the FP64 accumulators.
template <int D>
__device__ __forceinline__ void flush_path_grads(double (&dz)[D], double dval, int lane, double* g_slot_p,
                                                 double* g_val_p) {
#pragma unroll
    for (int j = 0; j <= D; ++j) {
        double x = j < D ? dz[j] : dval;
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
        if (lane == 0) {
            if (j < D) atomicAdd(&g_slot_p[j], x);
            else atomicAdd(g_val_p, x);
        }
    }
}

// ------------------------------------------------- two samples per lane --
//
// Tiles of 64 samples have rows of kTileLd2 floats; lane l owns columns 2l, 2l + 1.
constexpr int kTileLd2 = 66;

// 64-bit shared load that the compiler may not hoist out of the node loop
// (keeping all D pairs live would cost 2 D registers).
__device__ __forceinline__ float2 lds_pair(const float2* p) {
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(smem_u32(p)));
    return v;
}

// ------------------------------------------------------------------ FP64 --

template <int D, bool HAS_NAN>
__device__ __forceinline__ void bwd_path_f64(const Rec64* __restrict__ r, const float* __restrict__ xs,
                                             const float* __restrict__ gs, int lane, const QuadD& q,
                                             double* g_slot_p, double* g_val_p) {
    const double val = r[0].z;
    double dd[D], uu[D], acc1[D], acc2[D];
#pragma unroll
    for (int j = 0; j < D; ++j) {
        const Rec64 e = r[1 + j];
        const int f = feat_of(e.bits);
        const float x = xs[f * kTileLd + lane];
        const bool o = satisfies<HAS_NAN>(x, e.lo, e.hi, e.bits);
        dd[j] = (o ? 1.0 : 0.0) - e.z;
        uu[j] = (double)gs[f * kTileLd + lane] * dd[j];
        acc1[j] = acc2[j] = 0.0;
    }
    for (int m = 0; m < q.n; ++m) {
        const double t = q.t[m];
        double A[D], P[D], PU[D];
        P[0] = q.w[m];
        PU[0] = 0.0;
#pragma unroll
        for (int j = 0; j < D; ++j) {
            A[j] = fma(t, dd[j], r[1 + j].z);
            if (j + 1 < D) {
                P[j + 1] = P[j] * A[j];
                PU[j + 1] = fma(PU[j], A[j], uu[j] * P[j]);
            }
        }
        double S = 1.0, SU = 0.0;
#pragma unroll
        for (int j = D - 1; j >= 0; --j) {
            acc1[j] = fma(P[j], S, acc1[j]);
            acc2[j] = fma(1.0 - t, fma(P[j], SU, PU[j] * S), acc2[j]);
            SU = fma(SU, A[j], uu[j] * S);
            S *= A[j];
        }
    }
    double dval = 0.0, dz[D];
#pragma unroll
    for (int j = 0; j < D; ++j) {
        const int f = feat_of(r[1 + j].bits);
        dval = fma(uu[j], acc1[j], dval);
        dz[j] = val * (acc2[j] - (double)gs[f * kTileLd + lane] * acc1[j]);
    }
    flush_path_grads<D>(dz, dval, lane, g_slot_p, g_val_p);
}


}  // namespace qts
