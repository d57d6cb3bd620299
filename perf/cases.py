"""The calls whose speed this repository looks after, as a program makes them.

Models are random-split regression trees on independent N(0,1) features (the
shape of gradient-boosted ensembles: a split's threshold is a random quantile of
its node's box, rows are divided accordingly, a node stops at the depth limit
or at 5 rows), with leaf values and features of a regression model; samples
are N(0,1) rows, upstream gradients N(0,1).  The models of another seed are other
models (features, thresholds, leaf values) on trees of the same shape.

The FP32 tables give phi and the gradients to FP32 accuracy in float64 buffers
(their sums over paths are FP64); a program keeps them as float32 attributions or
parameter gradients, as QTreeShapFn does, so those runs end with that cast.  The
FP64 tables' results stay float64.
"""
import math
import random

import numpy as np
import torch

import paper_2605_04497_gb300 as qts

# ----------------------------------------------------------------- models --


class Model:
    """Node arrays of an ensemble as qts.Ensemble.from_arrays takes them."""

    def __init__(self, node_offsets, left, right, feature, threshold, default_left, z, leaf_value, n_features):
        self.node_offsets, self.left, self.right, self.feature = node_offsets, left, right, feature
        self.threshold, self.default_left, self.z, self.leaf_value = threshold, default_left, z, leaf_value
        self.n_features = n_features


def _grow(rng, shape, trees, depth, features, rows, leaf_std=0.1, full=False):
    """Level by level, all trees at once; `shape` draws how rows divide, `rng` the rest.  A node's box is known from its
    ancestors' splits: thresholds are drawn as quantiles of the feature's normal
    restricted to it, so the share of rows going left is the draw itself."""
    tree = np.arange(trees)
    n_rows = np.full(trees, rows, np.int64)
    af = np.full((trees, 0), -1, np.int32)      # ancestors' features
    lo_q = np.zeros((trees, 0))                 # and the quantile interval each edge leaves
    hi_q = np.ones((trees, 0))
    levels = []
    first = 0
    for level in range(depth + 1):
        n = len(tree)
        split = np.zeros(n, bool) if level == depth else (np.ones(n, bool) if full else n_rows > 5)
        f = rng.integers(0, features, n).astype(np.int32)
        u = shape.random(n) * 0.98 + 0.01
        same = af == f[:, None]
        lo = np.where(same, lo_q, 0.0).max(1, initial=0.0)
        hi = np.where(same, hi_q, 1.0).min(1, initial=1.0)
        q = lo + u * (hi - lo)
        thr = torch.special.ndtri(torch.from_numpy(np.clip(q, 1e-12, 1 - 1e-12))).numpy().astype(np.float32)
        nl = np.floor(u * n_rows).astype(np.int64)
        nr = n_rows - nl
        cl, cr = np.maximum(nl, 1), np.maximum(nr, 1)
        k = np.flatnonzero(split)
        left = np.full(n, -1, np.int64)
        left[k] = first + n + 2 * np.arange(len(k))
        levels.append(dict(tree=tree, left=left, feature=np.where(split, f, -1), thr=np.where(split, thr, 0),
                           dl=rng.integers(0, 2, n), zl=(cl / (cl + cr))[k], n_split=len(k)))
        if len(k) == 0:
            break
        two = np.repeat(k, 2)
        side = np.tile([0, 1], len(k))
        af = np.concatenate([af[two], f[two, None]], 1)
        lo_q = np.concatenate([lo_q[two], np.where(side == 0, 0.0, q[two])[:, None]], 1)
        hi_q = np.concatenate([hi_q[two], np.where(side == 0, q[two], 1.0)[:, None]], 1)
        n_rows = np.where(side == 0, nl[two], nr[two])
        tree = tree[two]
        first += n
    cat = lambda name: np.concatenate([v[name] for v in levels])
    tree, left, feature = cat("tree"), cat("left"), cat("feature")
    z = np.concatenate([np.ones(trees)] + [np.stack([v["zl"], 1 - v["zl"]], 1).ravel() for v in levels])
    # nodes grouped by tree; children become indices within their tree
    order = np.argsort(tree, kind="stable")
    offsets = np.concatenate([[0], np.cumsum(np.bincount(tree, minlength=trees))])
    new = np.empty(len(order), np.int64)
    new[order] = np.arange(len(order))
    local = new - offsets[tree]
    inner = left >= 0
    l = np.where(inner, local[np.where(inner, left, 0)], -1)
    r = np.where(inner, local[np.where(inner, left + 1, 0)], -1)
    leaf = np.where(inner, 0.0, rng.standard_normal(len(tree)) * leaf_std)
    g = lambda a, dt: np.ascontiguousarray(a[order], dtype=dt)
    return Model(offsets.astype(np.int64), g(l, np.int32), g(r, np.int32), g(feature, np.int32),
                 g(cat("thr"), np.float32), g(cat("dl"), np.uint8), g(z, np.float32), g(leaf, np.float32), features)


def _inputs(case, seed, i=0):
    """(model, X, grad_phi or None) of request i of a case, on the host."""
    rng = np.random.default_rng([seed, i])
    c = _request(case, i)
    model = _grow(rng, np.random.default_rng([c["trees"], c["depth"], i]), c["trees"], c["depth"], c["features"],
                  c["rows"], full=c["kind"] == "phi" and c["depth"] <= 4)
    X = rng.standard_normal((c["samples"], c["features"]), dtype=np.float32)
    if case.get("missing"):
        X[rng.random(X.shape, dtype=np.float32) < case["missing"]] = np.nan
    grad = None
    if c["kind"] in ("grad", "batch"):
        grad = rng.standard_normal((c["samples"], c["features"] + 1), dtype=np.float32)
    return model, X, grad


def _request(case, i):
    """A batch's requests have sizes of their own, spread over the case's ranges."""
    if case["kind"] != "batch":
        return case
    r = random.Random(case["spread"] * 1000 + i)
    part = lambda hi, lo: max(1, int(round(math.exp(r.uniform(math.log(lo), math.log(hi))))))
    depth = r.randint(3, case["depth"])
    return dict(kind="batch", trees=part(case["trees"], max(1, case["trees"] / 20)), depth=depth,
                features=part(case["features"], 8), samples=part(case["samples"], max(1, case["samples"] / 100)),
                rows=min(case["rows"], 20 * 2 ** depth))


# ------------------------------------------------------------------ cases --


def _case(name, kind, trees, depth, features, samples, rows, **more):
    c = dict(kind=kind, trees=trees, depth=depth, features=features, samples=samples, rows=rows, n_quad=8)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a small model on a handful of rows: launches and latency
        _case("phi-small", "phi", 10, 4, 8, 100, 1000),
        # one row of a served model, explained as it is asked for
        _case("phi-one-row", "phi", 300, 8, 50, 1, 100000),
        # attributions of a whole data set under a boosted ensemble: the main use
        _case("phi-boosted", "phi", 1000, 8, 50, 10000, 100000),
        # deep unpruned trees (features repeat along paths and merge)
        _case("phi-deep", "phi", 8, 20, 24, 5000, 200000),
        # an odd-sized data set with missing values, Thm 2's point counts
        _case("phi-missing", "phi", 300, 6, 31, 3001, 50000, missing=0.1, n_quad=qts.EXACT_NODES),
        # gradients of a loss on the attributions with respect to the model
        _case("grad-boosted", "grad", 200, 8, 50, 4001, 100000),
        # attributions and gradients of many models of different shapes at once
        _case("batch-mixed", "batch", 100, 14, 60, 4000, 100000, requests=8, spread=7),
        # the same for a service's small requests
        _case("batch-small", "batch", 60, 8, 40, 200, 5000, requests=16, spread=3),
        # pairwise interactions of a data set
        _case("pairs", "pairs", 500, 6, 30, 2000, 50000),
        # attributions in FP64, the mode results are checked with
        _case("phi-fp64", "phi", 50, 6, 13, 700, 20000, fp64=True),
    ]


def draw(rng):
    log = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    kind = rng.choice(["phi", "phi", "phi", "deep", "grad", "batch", "pairs", "fp64"])
    if kind == "phi":
        c = _case("", "phi", log(10, 1000), rng.randint(4, 10), log(8, 100), log(1, 10000), 100000)
        if rng.random() < 0.3:
            c["missing"] = 0.1
        if rng.random() < 0.3:
            c["n_quad"] = qts.EXACT_NODES
    elif kind == "deep":
        c = _case("", "phi", log(1, 8), rng.randint(11, 20), log(12, 60), log(100, 5000), 200000)
    elif kind == "grad":
        c = _case("", "grad", log(10, 400), rng.randint(4, 10), log(8, 100), log(50, 6000), 100000)
    elif kind == "batch":
        c = _case("", "batch", log(20, 100), rng.randint(6, 14), log(12, 80), log(100, 4000), 100000,
                  requests=rng.randint(2, 16), spread=rng.randint(0, 10 ** 6))
    elif kind == "pairs":
        c = _case("", "pairs", log(20, 500), rng.randint(3, 8), log(8, 60), log(50, 2000), 50000)
    else:
        c = _case("", "phi", log(5, 60), rng.randint(3, 7), log(8, 40), log(20, 900), 20000, fp64=True)
    # no drawn case costs more than the largest listed one
    while _ops(c) > 0.5 * _ops(listed()[2]) or (c.get("fp64") and _ops(c) > 2 * _ops(listed()[9])):
        c["samples"] = max(1, c["samples"] // 2)
        c["trees"] = max(1, c["trees"] * 2 // 3)
    return c


def _leaves(c):
    """About how many leaves a tree has: splits at random quantiles leave a tree
    full to depth 8 or so and thin it out below, down to a sixth of its rows."""
    return min(2.0 ** c["depth"] * min(1.0, 0.87 ** (c["depth"] - 8)), c["rows"] / 6.0)


def _ops(case):
    """FP operations of the method: per sample and split node and quadrature
    point, the depth-first form's edge factor, product, sum and dot of both edges;
    the adjoint carries derivatives along."""
    total = 0.0
    for i in range(case.get("requests", 1)):
        c = _request(case, i)
        nodes = c["trees"] * _leaves(c)
        points = 8 if case["n_quad"] else max(1, c["depth"] // 2)
        per = 7 * 2 * points
        if c["kind"] in ("grad", "batch"):
            per *= 3
        if c["kind"] == "pairs":
            per *= c["depth"] / 2
        total += nodes * per * c["samples"]
    return total


def work(case):
    total = 0.0
    for i in range(case.get("requests", 1)):
        c = _request(case, i)
        nodes = 2 * c["trees"] * _leaves(c)
        total += nodes * 20 + 4.0 * c["samples"] * c["features"]          # the model and the samples
        if c["kind"] == "pairs":
            total += 4.0 * c["samples"] * (c["features"] + 1) ** 2
        elif c["kind"] != "grad":
            total += 8.0 * c["samples"] * (c["features"] + 1)
        if c["kind"] in ("grad", "batch"):
            total += 4.0 * c["samples"] * (c["features"] + 1) + 16 * nodes
    return {"bytes": total, "flops": _ops(case)}


# -------------------------------------------------------------------- run --


def prepare(case, seed):
    if case["kind"] == "batch":
        return _prepare_batch(case, seed)
    model, X, grad = _inputs(case, seed)
    state = dict(case=case, ens=qts.Ensemble.from_arrays(model, fp64=bool(case.get("fp64"))),
                 X=torch.from_numpy(X).cuda())
    if grad is not None:
        state["grad"] = torch.from_numpy(grad).cuda()
    return state


def _prepare_batch(case, seed):
    """Requests of one batch; their results lie in one buffer, as a program that
    hands them on together lays them out."""
    items, n = [], 0
    for i in range(case["requests"]):
        model, X, grad = _inputs(case, seed, i)
        E = qts.Ensemble.from_arrays(model)
        M, F = X.shape
        items.append(dict(ens=E, X=torch.from_numpy(X).cuda(), grad_phi=torch.from_numpy(grad).cuda(),
                          at=n, shape=(M, F + 1)))
        n += M * (F + 1) + 2 * E.n_nodes
    out = torch.empty(n, dtype=torch.float64, device="cuda")
    for it in items:
        a, (M, C), N = it["at"], it["shape"], it["ens"].n_nodes
        it["phi"] = out[a:a + M * C].view(M, C)
        it["d_leaf"] = out[a + M * C:a + M * C + N]
        it["d_z"] = out[a + M * C + N:a + M * C + 2 * N]
    return dict(case=case, items=items, out=out, reqs=qts.make_requests(items))


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        qts.batched_fwd_bwd(state["reqs"], case["n_quad"])
        out = state["out"].float()
        got = {"phi": [], "d_leaf": [], "d_z": []}
        for it in state["items"]:
            a, (M, C), N = it["at"], it["shape"], it["ens"].n_nodes
            got["phi"].append(out[a:a + M * C].view(M, C))
            got["d_leaf"].append(out[a + M * C:a + M * C + N])
            got["d_z"].append(out[a + M * C + N:a + M * C + 2 * N])
        return got
    if case["kind"] == "grad":
        d_leaf, d_z = qts.shap_backward(state["ens"], state["X"], state["grad"], case["n_quad"])
        return {"d_leaf": d_leaf.float(), "d_z": d_z.float()}
    if case["kind"] == "pairs":
        return qts.shap_interactions(state["ens"], state["X"], case["n_quad"])
    phi = qts.shap_values(state["ens"], state["X"], case["n_quad"])
    return phi if case.get("fp64") else phi.float()


# ------------------------------------------------------------------ exact --


def _paths(m):
    """Every root-to-leaf path of a model, its splits merged per feature, grouped
    by the number d of features: (d, leaf, feature, lo, hi, nan_ok, z, edges) with
    [path, d] arrays and the edges as (path, element, node, product of the
    element's other edge weights)."""
    n = len(m.left)
    tree = np.repeat(np.arange(len(m.node_offsets) - 1), np.diff(m.node_offsets))
    base = m.node_offsets[tree]
    parent = np.full(n, -1, np.int64)
    side = np.zeros(n, np.int8)
    k = np.flatnonzero(m.left >= 0)
    for s, child in ((0, m.left), (1, m.right)):
        parent[base[k] + child[k]] = k
        side[base[k] + child[k]] = s
    leaf = np.flatnonzero(m.left < 0)
    depth = 0
    chain = []
    v = leaf
    while (parent[v] >= 0).any():
        chain.append(np.where(parent[v] >= 0, v, -1))
        v = np.where(parent[v] >= 0, parent[v], v)
        depth += 1
    L = len(leaf)
    feat = np.full((L, depth + 1), -1, np.int64)
    lo = np.full((L, depth + 1), -np.inf, np.float32)
    hi = np.full((L, depth + 1), np.inf, np.float32)
    ok = np.ones((L, depth + 1), bool)
    z = np.ones((L, depth + 1))
    d = np.zeros(L, np.int64)
    slot_of = []
    rows = np.arange(L)
    for c in reversed(chain):
        on = c >= 0
        p = np.where(on, parent[np.maximum(c, 0)], 0)
        f = m.feature[p]
        hit = feat == f[:, None]
        seen = hit.any(1)
        j = np.where(seen, hit.argmax(1), d)
        r = rows[on]
        jj = j[on]
        feat[r, jj] = f[on]
        w = m.z[c[on]].astype(np.float64)
        z[r, jj] *= w
        t, left = m.threshold[p[on]], side[c[on]] == 0
        hi[r, jj] = np.where(left, np.minimum(hi[r, jj], t), hi[r, jj])
        lo[r, jj] = np.where(left, lo[r, jj], np.maximum(lo[r, jj], t))
        ok[r, jj] &= (m.default_left[p[on]] != 0) == left
        d += on & ~seen
        slot_of.append((r, jj, c[on]))
    er = np.concatenate([s[0] for s in slot_of]) if slot_of else np.zeros(0, np.int64)
    ej = np.concatenate([s[1] for s in slot_of]) if slot_of else np.zeros(0, np.int64)
    en = np.concatenate([s[2] for s in slot_of]) if slot_of else np.zeros(0, np.int64)
    ec = z[er, ej] / m.z[en].astype(np.float64)
    out = []
    for width in np.unique(d):
        sel = np.flatnonzero(d == width)
        if width == 0:
            continue
        at = np.full(L, -1)
        at[sel] = np.arange(len(sel))
        e = at[er] >= 0
        w = slice(0, int(width))
        out.append((int(width), leaf[sel], feat[sel, w], lo[sel, w], hi[sel, w], ok[sel, w], z[sel, w],
                    (at[er[e]], ej[e], en[e], ec[e])))
    return out, leaf[d == 0]


def _rule(n_quad, width):
    """Gauss-Legendre points on [0, 1]: n_quad, or as few as are exact."""
    need = max(1, (width + 1) // 2)
    x, w = np.polynomial.legendre.leggauss(need if n_quad == 0 else min(n_quad, need))
    return [(0.5 * (a + 1), 0.5 * b) for a, b in zip(x, w)]


def _exact_one(model, X, grad, n_quad, pairs=False):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    M, F = X.shape
    x = torch.from_numpy(X).to(dev).t().contiguous()
    groups, bare = _paths(model)
    phi = torch.zeros(F + 1, M, dtype=torch.float64, device=dev)
    d_leaf = torch.zeros(len(model.left), dtype=torch.float64, device=dev)
    d_z = torch.zeros_like(d_leaf)
    sii = torch.zeros(F * F, M, dtype=torch.float64, device=dev) if pairs else None
    G = torch.from_numpy(grad).to(dev).double().t().contiguous() if grad is not None else None
    g_bias = G[F].sum() if grad is not None else None
    bias = float(model.leaf_value[bare].astype(np.float64).sum())
    if grad is not None and len(bare):
        d_leaf[torch.from_numpy(bare).to(dev)] = g_bias
    for width, leaf, feat, lo, hi, ok, z, (er, ej, en, ec) in groups:
        val_np = model.leaf_value[leaf].astype(np.float64)
        bias += float((val_np * z.prod(1)).sum())
        step = max(1, int(2e7 // max(1, M) // (3 if grad is not None else 1)))
        rule = _rule(n_quad, width)
        gz = torch.zeros(len(leaf), width, dtype=torch.float64, device=dev)
        gv = torch.zeros(len(leaf), dtype=torch.float64, device=dev)
        for a in range(0, len(leaf), step):
            s = slice(a, a + step)
            up = lambda v: torch.from_numpy(np.ascontiguousarray(v[s])).to(dev)
            ft, l, h, nk, zz, val = up(feat), up(lo), up(hi), up(ok), up(z), up(val_np)
            D, Z, U = [], [], []
            for j in range(width):
                xj = x[ft[:, j]]
                o = (xj >= l[:, j, None]) & (xj < h[:, j, None]) | (torch.isnan(xj) & nk[:, j, None])
                Z.append(zz[:, j, None])
                D.append(o.double() - Z[j])
                if grad is not None:
                    U.append(G[ft[:, j]] * D[j])
            acc = [torch.zeros_like(D[0]) for _ in range(width)]
            acc2 = [torch.zeros_like(D[0]) for _ in range(width)] if grad is not None else None
            pair = {}
            for t, w in rule:
                A = [torch.add(Z[j], D[j], alpha=t) for j in range(width)]
                P = [torch.full_like(D[0], w)]
                for j in range(width - 1):
                    P.append(P[j] * A[j])
                S = torch.ones_like(D[0])
                if grad is not None:
                    PU = [torch.zeros_like(D[0])]
                    for j in range(width - 1):
                        PU.append(PU[j] * A[j] + U[j] * P[j])
                    SU = torch.zeros_like(D[0])
                suffix = [None] * width
                for j in reversed(range(width)):
                    acc[j].addcmul_(P[j], S)
                    if grad is not None:
                        acc2[j].add_(torch.addcmul(PU[j] * S, P[j], SU), alpha=1 - t)
                        SU = torch.addcmul(U[j] * S, SU, A[j])
                    suffix[j] = S
                    S = S * A[j]
                if pairs:
                    for i in range(width):
                        R = P[i]
                        for j in range(i + 1, width):
                            term = R * suffix[j]
                            pair[i, j] = pair[i, j] + term if (i, j) in pair else term
                            R = R * A[j]
            for j in range(width):
                phi.index_add_(0, ft[:, j], acc[j] * D[j] * val[:, None])
                if grad is not None:
                    gv[s] += (U[j] * acc[j]).sum(1)
                    gz[s, j] = val * (acc2[j] - G[ft[:, j]] * acc[j]).sum(1)
            for (i, j), v in pair.items():
                v = v * D[i] * D[j] * val[:, None]
                sii.index_add_(0, ft[:, i] * F + ft[:, j], v)
                sii.index_add_(0, ft[:, j] * F + ft[:, i], v)
        if grad is not None:
            zt, vt = torch.from_numpy(z).to(dev), torch.from_numpy(val_np).to(dev)
            d_leaf[torch.from_numpy(leaf).to(dev)] = gv + g_bias * zt.prod(1)
            for j in range(width):
                gz[:, j] += g_bias * vt * torch.cat([zt[:, :j], zt[:, j + 1:]], 1).prod(1)
            on = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(dev)
            d_z.index_add_(0, on(en), gz[on(er), on(ej)] * on(ec))
    phi[F] = bias
    if pairs:
        half = 0.5 * sii.view(F, F, M).permute(2, 0, 1)
        full = torch.zeros(M, F + 1, F + 1, dtype=torch.float64, device=dev)
        full[:, :F, :F] = half
        i = torch.arange(F, device=dev)
        full[:, i, i] = phi[:F].t() - half.sum(2)
        full[:, F, F] = bias
        return full
    return phi.t().contiguous(), d_leaf, d_z


def exact(case, seed):
    with torch.no_grad():
        if case["kind"] == "batch":
            got = {"phi": [], "d_leaf": [], "d_z": []}
            for i in range(case["requests"]):
                phi, d_leaf, d_z = _exact_one(*_inputs(case, seed, i), case["n_quad"])
                for k, v in (("phi", phi), ("d_leaf", d_leaf), ("d_z", d_z)):
                    got[k].append(v)
            return got
        model, X, grad = _inputs(case, seed)
        if case["kind"] == "pairs":
            return _exact_one(model, X, None, case["n_quad"], pairs=True)
        phi, d_leaf, d_z = _exact_one(model, X, grad, case["n_quad"])
        return {"d_leaf": d_leaf, "d_z": d_z} if case["kind"] == "grad" else phi
