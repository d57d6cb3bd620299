// Host construction of the block tables (layout in qts_blocks.h): trees are
// walked in parallel, each thread appends to its own copy of every bucket, and
// the copies are joined in tree order.
#include "qts_blocks.h"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <thread>

#include "qts_threads.h"

namespace qts {

namespace {

struct Edge {
    int32_t feat;
    uint8_t went_left, def_left, is_cat;
    float thr;
    uint64_t cats;
    double w;
    int64_t child;
};

struct Elem {  // the splits on one feature along a path, merged (Eq. q_def)
    double z = 1.0;
    float lo = -INFINITY, hi = INFINITY;
    uint64_t cats = ~0ull;
    uint8_t nan_ok = 1, is_cat = 0, other_ok = 1;
};

Rec32 four(float a, float b, float c, float d) {
    Rec32 r{a, b, c, 0u};
    std::memcpy(&r.bits, &d, 4);
    return r;
}

constexpr int kKeys = (kMaxD + 1) * (kBlkMaxH + 1);

struct Part {  // one thread's share of one bucket
    std::vector<Rec32> rec;
    std::vector<double> dbl;
    std::vector<BlockEntry> ent;
    std::vector<uint32_t> ent_count;  // per block
    int64_t n = 0;
    int dmax = 0;
};

struct Walker {
    const qts_ensemble* e;
    bool grad;
    Part part[kKeys];
    std::vector<Edge> path;
    // per node of the current tree: unique features above it, whether its feature
    // is among them, the height of the block rooted at it (-1: none) and the least
    // cost of the subtree's blocks
    std::vector<int16_t> uniq;
    std::vector<uint8_t> rep;
    std::vector<int8_t> root;
    std::vector<double> best;
    std::vector<int32_t> order;
    std::vector<int32_t> count;  // per feature: edges of the walk's path that split on it
    int n_uniq = 0;              // features with count > 0
    std::vector<int> own;        // scratch of chain()
    std::vector<double> after;
    int64_t base = 0;

    // scratch of the block under construction
    std::vector<Rec32> rec;
    std::vector<double> dbl;
    std::vector<BlockEntry> ent;
    int H = 0, slot0 = 0, dmax = 0;  // slot0: the block's width
    bool fp64 = false;

    Edge edge(int64_t g, int side) const {
        const int32_t c = side == 0 ? e->left[g] : e->right[g];
        Edge x;
        x.feat = e->feature[g];
        x.went_left = side == 0;
        x.def_left = e->defl[g] != 0;
        x.is_cat = !e->is_cat.empty() && e->is_cat[g];
        x.cats = x.is_cat ? (side == 0 ? e->cat_left[g] : ~e->cat_left[g]) : ~0ull;
        x.thr = e->thr[g];
        x.w = (double)e->z[base + c];
        x.child = base + c;
        return x;
    }

    Elem merged(int32_t f) const {
        Elem m;
        for (const Edge& x : path) {
            if (x.feat != f) continue;
            m.z *= x.w;
            if (x.is_cat) {
                m.is_cat = 1;
                m.cats &= x.cats;
                if (x.went_left) m.other_ok = 0;
            } else if (x.went_left) {
                m.hi = std::min(m.hi, x.thr);
            } else {
                m.lo = std::max(m.lo, x.thr);
            }
            if (x.went_left != x.def_left) m.nan_ok = 0;
        }
        return m;
    }

    // {z, z, lo, hi} of the path's element on f, and its feature word
    Rec32 elem_rec(int32_t f, uint32_t* word) const {
        const Elem m = merged(f);
        *word = (uint32_t)f | (m.nan_ok ? kNanOk : 0u);
        if (!m.is_cat) return four((float)m.z, (float)m.z, m.lo, m.hi);
        const uint32_t l = (uint32_t)(m.cats & 0xFFFFFFFFull), h = (uint32_t)(m.cats >> 32);
        float lo, hi;
        std::memcpy(&lo, &l, 4);
        std::memcpy(&hi, &h, 4);
        *word |= kCat | (m.other_ok ? kOtherOk : 0u);
        return four((float)m.z, (float)m.z, lo, hi);
    }

    void add(int64_t node, bool leaf, int slot, double coef) {
        ent.push_back({(uint32_t)slot, ((uint32_t)node << 1) | (leaf ? 1u : 0u), coef});
    }

    // chain the z-gradient in `slot` (times scale) of the path's element on f to
    // its edges: dz/dw = product of the element's other edge weights
    void chain(int32_t f, int slot, double scale) {
        own.clear();
        for (size_t k = 0; k < path.size(); ++k)
            if (path[k].feat == f) own.push_back((int)k);
        if (own.size() <= 8) {
            for (int a : own) {
                double c = scale;
                for (int b : own)
                    if (b != a) c *= path[b].w;
                add(path[a].child, false, slot, c);
            }
            return;
        }
        // long chains (degenerate trees): products before and after each edge
        after.assign(own.size() + 1, 1.0);
        for (size_t k = own.size(); k-- > 0;) after[k] = after[k + 1] * path[own[k]].w;
        double before = scale;
        for (size_t k = 0; k < own.size(); ++k) {
            add(path[own[k]].child, false, slot, before * after[k + 1]);
            before *= path[own[k]].w;
        }
    }

    bool is_leaf(int32_t v) const { return e->left[base + v] < 0; }
    // may v be a node of a block below its root
    bool inside(int32_t v) const { return !rep[v] && (e->is_cat.empty() || !e->is_cat[base + v]); }

    // least cost of what a block leaves out below u, `levels` levels of splits
    // still being available to it there
    double outside(int32_t u, int levels) const {
        if (is_leaf(u)) return 0.0;
        if (levels == 0 || !inside(u)) return best[u];
        return outside(e->left[base + u], levels - 1) + outside(e->right[base + u], levels - 1);
    }

    Rec32 word_rec(int32_t f, float thr, float lo, float hi, bool nan_ok, bool def_left) const {
        return {thr, lo, hi, (uint32_t)f | (nan_ok ? kNanOk : 0u) | (def_left ? kDefLeft : 0u)};
    }

    // Lay out the tree node v (-1: an empty leaf) as node n; `levels` levels
    // below and including n.
    void place(int32_t v, int n, int levels) {
        Rec32* r = &rec[blk_rec(H, n)];
        const int slot = slot0 + blk_slot(H, n);
        const bool split = v >= 0 && !is_leaf(v) && (n == 1 || inside(v));
        if (!split) {
            // neutral; a leaf goes down the left edges to a pair's left leaf
            const bool leaf = v >= 0 && is_leaf(v);
            const float val = leaf ? e->leaf[base + v] : 0.f;
            double* q = &dbl[blk_dbl(slot0, H, n)];
            r[1] = word_rec(e->n_features, INFINITY, -INFINITY, INFINITY, true, true);
            if (levels > 1) {
                r[0] = four(1.f, 1.f, 0.f, 0.f);
                q[0] = 1.0;
                q[1] = 0.0;
                place(leaf ? v : -1, 2 * n, levels - 1);
                place(-1, 2 * n + 1, levels - 1);
            } else {
                r[0] = four(val, 0.f, 1.f, 0.f);
                r[2] = four(val, val, 0.f, 0.f);
                q[0] = q[4] = val;
                q[1] = q[3] = 0.0;
                q[2] = 1.0;
                if (leaf) {
                    dmax = std::max(dmax, (int)uniq[v]);
                    if (grad) {
                        add(base + v, true, slot, 1.0);
                        add(base + v, true, slot + 1, 1.0);
                    }
                }
            }
            return;
        }
        const int64_t g = base + v;
        const int32_t f = e->feature[g];
        const Elem prev = merged(f);
        r[1] = word_rec(f, e->thr[g], prev.lo, prev.hi, prev.nan_ok != 0, e->defl[g] != 0);
        float z[2], val[2] = {0.f, 0.f};
        double zd[2], vz = 0.0;
        for (int side = 0; side < 2; ++side) {
            const Edge x = edge(g, side);
            const int32_t c = (int32_t)(x.child - base);
            const double ze = prev.z * x.w;
            z[side] = (float)ze;
            zd[side] = ze;
            path.push_back(x);
            if (levels > 1) {
                if (grad) chain(f, slot + side, 1.0);
                place(c, 2 * n + side, levels - 1);
            } else if (is_leaf(c)) {
                val[side] = e->leaf[x.child];
                vz += (double)val[side] * ze;
                dmax = std::max(dmax, (int)uniq[c]);
                if (grad) {
                    add(x.child, true, slot, ze);
                    add(x.child, true, slot + 1 + side, 1.0);
                    chain(f, slot, (double)val[side]);
                }
            }
            path.pop_back();
        }
        double* q = &dbl[blk_dbl(slot0, H, n)];
        if (levels > 1) {
            r[0] = four(z[0], z[0], z[1], z[1]);
            q[0] = zd[0];
            q[1] = zd[1];
        } else {
            r[0] = four(val[0], val[1], z[0], z[1]);
            r[2] = four((float)vz, (float)vz, 0.f, 0.f);
            q[0] = val[0];
            q[1] = val[1];
            q[2] = zd[0];
            q[3] = zd[1];
            q[4] = vz;
        }
    }

    void emit(int32_t v, int h) {
        const int64_t g = base + v;
        H = h;
        int32_t pre[kMaxD];
        int D = 0;
        for (const Edge& x : path)
            if (!(h > 0 && x.feat == e->feature[g]) && std::find(pre, pre + D, x.feat) == pre + D) pre[D++] = x.feat;
        const int width = D == 0 ? 0 : bucket_width_for(D);
        slot0 = width;
        dmax = h == 0 ? uniq[v] : 0;
        ent.clear();
        rec.resize((size_t)(blk_stride(0, h) - blk_head(0)));
        dbl.assign((size_t)blk_doubles(width, h), 1.0);
        dbl[0] = h == 0 ? (double)e->leaf[g] : 1.0;
        for (int j = 0; j < D; ++j) dbl[1 + j] = merged(pre[j]).z;
        if (h > 0) place(v, 1, h);
        Part& P = part[width * (kBlkMaxH + 1) + h];
        P.rec.push_back(four(h == 0 ? e->leaf[g] : 1.f, 0.f, 0.f, 0.f));
        uint32_t word[kMaxD + 3];
        for (int j = 0; j < (width + 3) / 4 * 4; ++j) {
            // padding: a neutral element on the tile's zero row
            Rec32 r = four(1.f, 1.f, -INFINITY, INFINITY);
            word[j] = (uint32_t)e->n_features | kNanOk;
            if (j < D) r = elem_rec(pre[j], &word[j]);
            if (j < width) P.rec.push_back(r);
        }
        for (int j = 0; j < width; j += 4) {
            Rec32 r;
            std::memcpy(&r, &word[j], sizeof(r));
            P.rec.push_back(r);
        }
        P.rec.insert(P.rec.end(), rec.begin(), rec.end());
        if (fp64) P.dbl.insert(P.dbl.end(), dbl.begin(), dbl.end());
        if (grad) {
            for (int j = 0; j < D; ++j) chain(pre[j], j, 1.0);
            if (h == 0) add(g, true, slot0, 1.0);
            P.ent.insert(P.ent.end(), ent.begin(), ent.end());
            P.ent_count.push_back((uint32_t)ent.size());
        }
        P.dmax = std::max(P.dmax, dmax);
        ++P.n;
    }

    // Visit the nodes with their paths: on(v) returns whether to go on below v.
    template <typename On>
    void walk(const On& on) {
        struct Item { int32_t v; int32_t depth; Edge in; };
        std::vector<Item> stack;
        stack.push_back({0, 0, {}});
        path.clear();
        count.assign((size_t)e->n_features, 0);
        n_uniq = 0;
        while (!stack.empty()) {
            const Item it = stack.back();
            stack.pop_back();
            for (; (int)path.size() > std::max(0, it.depth - 1); path.pop_back())
                if (--count[path.back().feat] == 0) --n_uniq;
            if (it.depth > 0) {
                path.push_back(it.in);
                if (count[it.in.feat]++ == 0) ++n_uniq;
            }
            on(it.v);
            if (is_leaf(it.v)) continue;
            for (int side = 1; side >= 0; --side) {
                const Edge x = edge(base + it.v, side);
                stack.push_back({(int32_t)(x.child - base), it.depth + 1, x});
            }
        }
    }

    void tree(int t) {
        base = e->off[t];
        const int32_t n = (int32_t)(e->off[t + 1] - base);
        if (is_leaf(0)) return;  // no split: part of E[f] only
        uniq.assign((size_t)n, 0);
        rep.assign((size_t)n, 0);
        root.assign((size_t)n, -1);
        best.assign((size_t)n, 0.0);
        order.clear();
        walk([&](int32_t v) {
            order.push_back(v);
            uniq[v] = (int16_t)n_uniq;
            rep[v] = !is_leaf(v) && count[e->feature[base + v]] > 0;
        });
        // children come after their parents in `order`
        for (size_t i = order.size(); i-- > 0;) {
            const int32_t v = order[i];
            if (is_leaf(v)) {
                best[v] = blk_cost(bucket_width_for(std::max<int>(uniq[v], 1)), 0);
                continue;
            }
            const int32_t l = e->left[base + v], r = e->right[base + v];
            best[v] = best[l] + best[r];
            if (!e->is_cat.empty() && e->is_cat[base + v]) continue;
            const int D = uniq[v] - (rep[v] ? 1 : 0), W = D == 0 ? 0 : bucket_width_for(D);
            for (int h = 1; h <= blk_max_h(W); ++h) {
                const double c = blk_cost(W, h) + outside(l, h - 1) + outside(r, h - 1);
                if (c < best[v]) {
                    best[v] = c;
                    root[v] = (int8_t)h;
                }
            }
        }
        // the blocks in use: from the root down, a node is part of the block above
        // it, the root of one of its own, or between blocks
        std::vector<int32_t> todo(1, 0);
        std::vector<uint8_t> starts((size_t)n, 0);
        while (!todo.empty()) {
            const int32_t v = todo.back();
            todo.pop_back();
            if (is_leaf(v)) {
                starts[v] = 1;
                continue;
            }
            const int32_t l = e->left[base + v], r = e->right[base + v];
            if (root[v] < 0) {
                todo.push_back(l);
                todo.push_back(r);
                continue;
            }
            starts[v] = 1;
            cut(l, root[v] - 1, &todo);
            cut(r, root[v] - 1, &todo);
        }
        walk([&](int32_t v) {
            if (starts[v]) emit(v, is_leaf(v) ? 0 : root[v]);
        });
    }

    void cut(int32_t u, int levels, std::vector<int32_t>* todo) const {
        if (is_leaf(u)) return;
        if (levels == 0 || !inside(u)) {
            todo->push_back(u);
            return;
        }
        cut(e->left[base + u], levels - 1, todo);
        cut(e->right[base + u], levels - 1, todo);
    }
};

}  // namespace

void build_blocks(const qts_ensemble* e, bool grad, BlockHost* out) {
    const int64_t nodes = e->n_nodes;
    const unsigned hw = std::max(1u, std::thread::hardware_concurrency());
    const int nth = (int)std::max<int64_t>(
        1, std::min<int64_t>({(int64_t)hw, (int64_t)e->n_trees, std::max<int64_t>(1, nodes / 8000)}));
    std::vector<Walker> w((size_t)nth);
    std::vector<int> cut((size_t)nth + 1, e->n_trees);
    cut[0] = 0;
    for (int k = 1, t = 0; k < nth; ++k) {
        while (t < e->n_trees && e->off[t] < nodes * k / nth) ++t;
        cut[k] = std::max(cut[k - 1], t);
    }
    run_threads(nth, [&](int k) {
        w[k].e = e;
        w[k].grad = grad;
        w[k].fp64 = (e->flags & QTS_FLAG_FP64) != 0;
        for (int t = cut[k]; t < cut[k + 1]; ++t) w[k].tree(t);
    });
    // bucket sizes and each thread's place in them
    *out = BlockHost();
    int64_t n_rec = 0, n_dbl = 0, n_ent = 0, n_slot = 0, n_blk = 0;
    struct Place { int64_t rec, dbl, ent, slot; };
    std::vector<Place> at((size_t)nth * kKeys);
    for (int key = 0; key < kKeys; ++key) {
        BlockBucket b;
        b.D = key / (kBlkMaxH + 1);
        b.h = key % (kBlkMaxH + 1);
        b.rec_off = n_rec;
        b.dbl_off = n_dbl;
        b.slot_off = n_slot;
        for (int k = 0; k < nth; ++k) {
            const Part& p = w[k].part[key];
            at[(size_t)k * kKeys + key] = {n_rec, n_dbl, n_ent, n_slot + b.n * (b.D + blk_slots(b.h))};
            n_rec += (int64_t)p.rec.size();
            n_dbl += (int64_t)p.dbl.size();
            n_ent += (int64_t)p.ent.size();
            b.n += p.n;
            b.dmax = std::max(b.dmax, p.dmax);
        }
        if (b.n == 0) continue;
        n_slot += b.n * (b.D + blk_slots(b.h));
        n_blk += b.n;
        out->buckets.push_back(b);
    }
    out->n_blocks = n_blk;
    out->n_slots = n_slot;
    out->rec.resize((size_t)n_rec);
    out->dbl.resize((size_t)n_dbl);
    if (grad) {
        out->ent.resize((size_t)n_ent);
    }
    run_threads(nth, [&](int k) {
        for (int key = 0; key < kKeys; ++key) {
            const Part& p = w[k].part[key];
            const Place& a = at[(size_t)k * kKeys + key];
            if (p.n == 0) continue;
            std::memcpy(out->rec.data() + a.rec, p.rec.data(), p.rec.size() * sizeof(Rec32));
            if (!p.dbl.empty()) std::memcpy(out->dbl.data() + a.dbl, p.dbl.data(), p.dbl.size() * sizeof(double));
            if (!grad) continue;
            const int64_t stride = key / (kBlkMaxH + 1) + blk_slots(key % (kBlkMaxH + 1));
            const BlockEntry* src = p.ent.data();
            BlockEntry* dst = out->ent.data() + a.ent;
            for (int64_t i = 0; i < p.n; ++i)
                for (uint32_t k = 0; k < p.ent_count[(size_t)i]; ++k, ++src, ++dst) {
                    *dst = *src;
                    dst->slot += (uint32_t)(a.slot + i * stride);
                }
        }
    });
    if (!grad) return;
    // weights of G = sum_s grad_phi[s, F] in the gradients: E[f] = sum over leaves
    // of val times the edge weights above, so dE/dval is the leaf's reach and
    // dE/dw_c the reach of c's parent times the expectation below c
    out->bias_leaf.assign((size_t)nodes, 0.0);
    out->bias_z.assign((size_t)nodes, 0.0);
    run_threads(nth, [&](int k) {
        std::vector<int32_t> order;
        std::vector<double> reach, below;
        for (int t = cut[k]; t < cut[k + 1]; ++t) {
            const int64_t base = e->off[t];
            const size_t n = (size_t)(e->off[t + 1] - base);
            order.assign(1, 0);
            reach.assign(n, 1.0);
            below.assign(n, 0.0);
            for (size_t i = 0; i < order.size(); ++i) {
                const int32_t v = order[i];
                const int64_t g = base + v;
                if (e->left[g] < 0) {
                    below[v] = (double)e->leaf[g];
                    out->bias_leaf[g] = reach[v];
                    continue;
                }
                for (int32_t c : {e->left[g], e->right[g]}) {
                    reach[c] = reach[v] * (double)e->z[base + c];
                    order.push_back(c);
                }
            }
            for (size_t i = order.size(); i-- > 0;) {
                const int32_t v = order[i];
                const int64_t g = base + v;
                if (e->left[g] < 0) continue;
                for (int32_t c : {e->left[g], e->right[g]}) {
                    below[v] += (double)e->z[base + c] * below[c];
                    out->bias_z[base + c] = reach[v] * below[c];
                }
            }
        }
    });
}

}  // namespace qts
