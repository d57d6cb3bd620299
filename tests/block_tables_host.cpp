// Host evaluation of the block tables, for tests without a GPU: the tables as the
// library builds them, with the definitions at the head of qts_blocks.h in FP64, one
// sample, block and quadrature node at a time.
#include <atomic>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>

#include "qts_blocks.h"

// operator new that fails from the n-th allocation on (n < 0: never)
static std::atomic<long> g_allowed{-1};
void* operator new(size_t n) {
    if (g_allowed.load() >= 0 && g_allowed.fetch_sub(1) <= 0) {
        g_allowed.store(0);
        throw std::bad_alloc();
    }
    if (void* p = std::malloc(n ? n : 1)) return p;
    throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, size_t) noexcept { std::free(p); }

using namespace qts;

struct Tables {
    qts_ensemble e;
    BlockHost H;
};

namespace {

struct Sample {
    const float* x;
    const float* g;  // grad_phi row
    int F;
    float at(int f) const { return f < F ? x[f] : 0.f; }
    double grad(int f) const { return f < F ? (double)g[f] : 0.0; }
};

int feat(uint32_t w) { return (int)(w & kFeatMask); }
float as_float(uint32_t b) {
    float v;
    std::memcpy(&v, &b, 4);
    return v;
}
uint32_t as_bits(float v) {
    uint32_t b;
    std::memcpy(&b, &v, 4);
    return b;
}

bool satisfied(float x, float lo, float hi, uint32_t w) {
    if (x != x) return (w & kNanOk) != 0;
    if (!(w & kCat)) return x >= lo && x < hi;
    if (!(x >= 0.f && x < 64.f)) return (w & kOtherOk) != 0;
    const int c = (int)x;
    return (as_bits(c < 32 ? lo : hi) >> (c & 31)) & 1u;
}

// One block of one sample: contributions to phi and to the block's adjoint sums.
struct Block {
    int D, h;
    const Rec32* r;
    const double* dbl;  // FP64 weights, or nullptr: those of the records
    Sample s;
    double* phi;
    double* slots;
    double t = 0;

    struct Node {
        int f;
        double d[2], z[2], val[2], g, vd, vz;
        bool o[2];
    };
    Node node(int n) const {
        const Rec32* q = r + blk_head(D) + blk_rec(h, n);
        const bool pair = n > blk_inner(h);
        Node v;
        v.f = feat(q[1].bits);
        const float x = s.at(v.f);
        bool in = n == 1 ? x >= q[1].lo && x < q[1].hi : x < q[1].hi, left = x < q[1].z;
        if (x != x) {
            in = n != 1 || (q[1].bits & kNanOk);
            left = (q[1].bits & kDefLeft) != 0;
        }
        v.o[0] = in && left;
        v.o[1] = in && !left;
        const double* z64 = dbl ? dbl + blk_dbl(D, h, n) : nullptr;
        for (int k = 0; k < 2; ++k) {
            v.z[k] = pair ? (k ? as_float(q[0].bits) : q[0].hi) : (k ? q[0].hi : q[0].z);
            v.val[k] = pair ? (k ? q[0].lo : q[0].z) : 0.0;
            if (z64) v.z[k] = z64[pair ? 2 + k : k];
            if (z64 && pair) v.val[k] = z64[k];
            v.d[k] = (v.o[k] ? 1.0 : 0.0) - v.z[k];
        }
        v.vd = v.val[0] * v.d[0] + v.val[1] * v.d[1];
        v.vz = !pair ? 0.0 : z64 ? z64[4] : q[2].z;
        v.g = s.grad(v.f);
        return v;
    }

    // below node n, `levels` of splits; (C, CU): the product of the factors above and
    // its derivative along u = g d; returns the leaf sum and its derivative
    void down(int n, int levels, double C, double CU, double* G, double* GU) {
        const Node v = node(n);
        double* o = slots + D + blk_slot(h, n);
        if (levels == 1) {
            *G = v.vz + t * v.vd;
            *GU = v.g * v.vd;
            phi[v.f] += v.vd * C;
            const double q = (1.0 - t) * CU - v.g * C;
            o[0] += q;
            for (int k = 0; k < 2; ++k)
                if (v.o[k]) o[1 + k] += CU - q;
            return;
        }
        *G = *GU = 0.0;
        for (int k = 0; k < 2; ++k) {
            const double a = v.z[k] + t * v.d[k], u = v.g * v.d[k];
            double g, gu;
            down(2 * n + k, levels - 1, C * a, CU * a + u * C, &g, &gu);
            *G += a * g;
            *GU += a * gu + u * g;
            phi[v.f] += v.d[k] * C * g;
            o[k] += (1.0 - t) * (C * gu + CU * g) - v.g * C * g;
        }
    }

    void add(double tm, double w) {
        t = tm;
        const uint32_t* words = (const uint32_t*)(r + 1 + D);
        std::vector<double> a(D), d(D), g(D);
        double C = w, CU = 0.0, G, GU = 0.0;
        for (int j = 0; j < D; ++j) {
            const double z = dbl ? dbl[1 + j] : r[1 + j].z;
            const int f = feat(words[j]);
            d[j] = (satisfied(s.at(f), r[1 + j].hi, as_float(r[1 + j].bits), words[j]) ? 1.0 : 0.0) - z;
            a[j] = z + t * d[j];
            g[j] = s.grad(f);
            CU = CU * a[j] + g[j] * d[j] * C;
            C *= a[j];
        }
        if (h > 0) {
            down(1, h, C, CU, &G, &GU);
        } else {
            G = dbl ? dbl[0] : r[0].z;
            slots[D] += CU;
        }
        for (int j = 0; j < D; ++j) {  // the others' product and its derivative
            double R = w, RU = 0.0;
            for (int l = 0; l < D; ++l) {
                if (l == j) continue;
                RU = RU * a[l] + g[l] * d[l] * R;
                R *= a[l];
            }
            phi[feat(words[j])] += d[j] * R * G;
            slots[j] += (1.0 - t) * (R * GU + RU * G) - g[j] * R * G;
        }
    }
};

}  // namespace

extern "C" {

Tables* bt_new(int32_t n_trees, const int64_t* off, const int32_t* left, const int32_t* right, const int32_t* feature,
               const float* thr, const uint8_t* defl, const float* z, const float* leaf, const uint8_t* is_cat,
               const uint64_t* cat_left, int32_t F, int32_t fp64) {
    auto* T = new Tables();
    qts_ensemble& e = T->e;
    const int64_t N = off[n_trees];
    e.n_trees = n_trees;
    e.n_features = F;
    e.n_nodes = N;
    e.flags = fp64 ? QTS_FLAG_FP64 : 0u;
    e.off.assign(off, off + n_trees + 1);
    e.left.assign(left, left + N);
    e.right.assign(right, right + N);
    e.feature.assign(feature, feature + N);
    e.thr.assign(thr, thr + N);
    e.defl.assign(defl, defl + N);
    e.z.assign(z, z + N);
    e.leaf.assign(leaf, leaf + N);
    if (is_cat) {
        e.is_cat.assign(is_cat, is_cat + N);
        e.cat_left.assign(cat_left, cat_left + N);
    }
    return T;
}

void bt_free(Tables* T) { delete T; }

// 0, or 1 when memory ran out (allowed: allocations before every further one fails)
int32_t bt_build(Tables* T, int32_t grad, int64_t allowed) {
    g_allowed.store((long)allowed);
    int32_t rc = 0;
    try {
        build_blocks(&T->e, grad != 0, &T->H);
    } catch (const std::bad_alloc&) {
        rc = 1;
    }
    g_allowed.store(-1);
    return rc;
}

int32_t bt_prepare(Tables* T, int64_t allowed) {
    g_allowed.store((long)allowed);
    int32_t rc = 0;
    try {
        Prepared P;
        std::string err;
        qts_ensemble& e = T->e;
        const bool cat = !e.is_cat.empty();
        if (prepare(e.n_trees, e.off.data(), e.left.data(), e.right.data(), e.feature.data(), e.thr.data(),
                    e.defl.data(), e.z.data(), e.leaf.data(), cat ? e.is_cat.data() : nullptr,
                    cat ? e.cat_left.data() : nullptr, e.n_features, false, &P, &err) != QTS_OK)
            rc = 2;
    } catch (const std::bad_alloc&) {
        rc = 1;
    }
    g_allowed.store(-1);
    return rc;
}

int64_t bt_blocks(const Tables* T, int32_t h) {
    int64_t n = 0;
    for (const BlockBucket& b : T->H.buckets)
        if (b.h == h) n += b.n;
    return n;
}

// phi [M][F + 1] (column F is left alone but for padding's zeros) and the gradients
// of sum grad * phi without E[f]'s part
void bt_eval(const Tables* T, const float* X, const float* grad, int64_t M, int32_t n_quad, double* phi,
             double* d_leaf, double* d_z) {
    const int F = T->e.n_features;
    std::vector<double> tq(QTS_MAX_QUAD), wq(QTS_MAX_QUAD), slots((size_t)T->H.n_slots, 0.0);
    gauss_legendre(n_quad, tq.data(), wq.data());
    const bool fp64 = !T->H.dbl.empty();
    for (const BlockBucket& b : T->H.buckets) {
        const int ns = b.D + blk_slots(b.h);
        for (int64_t p = 0; p < b.n; ++p)
            for (int64_t s = 0; s < M; ++s) {
                Block k{b.D, b.h, T->H.rec.data() + b.rec_off + p * blk_stride(b.D, b.h),
                        fp64 ? T->H.dbl.data() + b.dbl_off + p * blk_doubles(b.D, b.h) : nullptr,
                        {X + s * F, grad + s * (F + 1), F}, phi + s * (F + 1), slots.data() + b.slot_off + p * ns};
                for (int m = 0; m < n_quad; ++m) k.add(tq[m], wq[m]);
            }
    }
    for (const BlockEntry& e : T->H.ent) ((e.target & 1u) ? d_leaf : d_z)[e.target >> 1] += e.coef * slots[e.slot];
}

void bt_bias(const Tables* T, double* bias_leaf, double* bias_z) {
    std::memcpy(bias_leaf, T->H.bias_leaf.data(), T->H.bias_leaf.size() * sizeof(double));
    std::memcpy(bias_z, T->H.bias_z.data(), T->H.bias_z.size() * sizeof(double));
}

}  // extern "C"
