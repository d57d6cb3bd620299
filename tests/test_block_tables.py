"""Block tables on the host (no GPU): records, weights, adjoint sums and their
entries, evaluated in FP64 by tests/block_tables_host.cpp, against the oracle on the
forms a tree can take: leaves at any height, features repeated at a block's root
and below it, chains, categorical splits, missing values and infinities.

The same host code checks that running out of memory while tables are built is an
error of the call, on whichever thread it happens."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
import synth
from helpers import caterpillar_ensemble, categorical_ensemble, rel_err_rows, tiny_ensemble

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_04497_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


@pytest.fixture(scope="session")
def host_lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("blocks") / "libblocks.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-pthread", "-Wl,-Bsymbolic", "-I", CSRC, "-I",
                    os.path.join(ROOT, "include"), "-I", os.path.join(CUDA, "include"), "-o", out,
                    os.path.join(ROOT, "tests", "block_tables_host.cpp"), os.path.join(CSRC, "qts_blocks.cpp"),
                    os.path.join(CSRC, "qts_prep.cpp")], check=True)
    return out


def load(path):
    L = ctypes.CDLL(path)
    vp, i32, i64 = ctypes.c_void_p, ctypes.c_int32, ctypes.c_int64
    L.bt_new.restype = vp
    L.bt_new.argtypes = [i32] + [vp] * 10 + [i32, i32]
    L.bt_free.argtypes = [vp]
    L.bt_build.argtypes = [vp, i32, i64]
    L.bt_prepare.argtypes = [vp, i64]
    L.bt_blocks.argtypes = [vp, i32]
    L.bt_blocks.restype = i64
    L.bt_eval.argtypes = [vp, vp, vp, i64, i32, vp, vp, vp]
    L.bt_eval.restype = None
    L.bt_bias.argtypes = [vp, vp, vp]
    L.bt_bias.restype = None
    return L


def tables(L, ens, fp64=False):
    arr = lambda a, dt: None if a is None else np.ascontiguousarray(a, dtype=dt)
    a = [arr(ens.node_offsets, np.int64), arr(ens.left, np.int32), arr(ens.right, np.int32),
         arr(ens.feature, np.int32), arr(ens.threshold, np.float32), arr(ens.default_left, np.uint8),
         arr(ens.z, np.float32), arr(ens.leaf_value, np.float32), arr(getattr(ens, "is_cat", None), np.uint8),
         arr(getattr(ens, "cat_left", None), np.uint64)]
    p = [None if x is None else x.ctypes.data for x in a]
    return L.bt_new(ens.n_trees, *p, ens.n_features, int(fp64))


def _chain(seed, depth, F):
    """One tree, a chain of `depth` splits over F features: every split repeats one."""
    ens = caterpillar_ensemble(seed, [depth], depth)
    ens.feature[:] = ens.feature % F
    ens.n_features = F
    return ens


CASES = {
    "one-split": lambda: synth.grow(1, 3, 1, 3, 50, 1.0, min_rows=2, full_depth=True),
    "full-2": lambda: synth.grow(2, 2, 2, 5, 100, 1.0, min_rows=2, full_depth=True),
    "full-3": lambda: synth.grow(3, 2, 3, 9, 200, 1.0, min_rows=2, full_depth=True),
    "ragged": lambda: tiny_ensemble(4, n_trees=4, depth=6, F=12),
    "repeats": lambda: tiny_ensemble(5, n_trees=3, depth=9, F=4, n_train=400),
    "two-features": lambda: tiny_ensemble(6, n_trees=3, depth=8, F=2, n_train=300),
    "one-feature": lambda: tiny_ensemble(7, n_trees=2, depth=6, F=1),
    "single-leaves": lambda: synth.concat([tiny_ensemble(8, n_trees=1, depth=3), tiny_ensemble(9, 1, 0)]),
    "chain": lambda: _chain(10, 24, 5),
    "wide-20": lambda: caterpillar_ensemble(11, [20, 9, 3], 24),
    "wide-41": lambda: caterpillar_ensemble(12, [41], 44),
    "categories": lambda: categorical_ensemble(13),
    "categories-deep": lambda: categorical_ensemble(14, depth=9, F=4, cat_features=(0, 1, 3)),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("fp64", [False, True])
def test_tables_against_the_oracle(host_lib, name, fp64):
    L = load(host_lib)
    ens = CASES[name]()
    F, M = ens.n_features, 24
    X = synth.normal(40, synth.STREAM_X, (M, F))
    cat = getattr(ens, "is_cat", None) is not None
    if cat:
        X = synth.categorical_columns(X, [f for f in range(F) if ens.is_cat[ens.feature == f].any()], 6, 41)
    r = np.random.default_rng(42)
    X[r.random(X.shape) < 0.1] = np.nan
    G = synth.normal(40, synth.STREAM_GRAD, (M, F + 1))
    T = tables(L, ens, fp64)
    assert L.bt_build(T, 1, -1) == 0
    phi = np.zeros((M, F + 1))
    d_leaf, d_z = np.zeros(ens.n_nodes), np.zeros(ens.n_nodes)
    L.bt_eval(T, X.ctypes.data, G.ctypes.data, M, 22, phi.ctypes.data, d_leaf.ctypes.data, d_z.ctypes.data)
    b_leaf, b_z = np.empty(ens.n_nodes), np.empty(ens.n_nodes)
    L.bt_bias(T, b_leaf.ctypes.data, b_z.ctypes.data)
    total = G[:, F].astype(np.float64).sum()
    ref = oracle.shap_exact(ens, X)
    dl_ref, dz_ref = oracle.grad_exact(ens, X, G)
    phi[:, F] = ref[:, F]
    # 22 points are exact for these widths: what is left is the weights' rounding, to FP32
    # (half an ulp each, up to 41 factors) or not at all
    tol = 1e-11 if fp64 else 42 * 6e-8
    assert rel_err_rows(phi, ref).max() <= tol
    rel = lambda a, b: np.abs(a - b).max() / max(np.abs(b).max(), 1e-300)
    assert rel(d_leaf + total * b_leaf, dl_ref) <= tol
    assert rel(d_z + total * b_z, dz_ref) <= tol
    L.bt_free(T)


def test_infinities(host_lib):
    """x = +-inf takes the sides that the half-open intervals of the splits give it."""
    L = load(host_lib)
    ens = tiny_ensemble(20, n_trees=3, depth=6, F=5)
    r = np.random.default_rng(20)
    X = synth.normal(43, synth.STREAM_X, (32, 5))
    u = r.random(X.shape)
    X[u < 0.2], X[(u >= 0.2) & (u < 0.4)] = np.inf, -np.inf
    G = np.zeros((32, 6), np.float32)
    T = tables(L, ens, True)
    assert L.bt_build(T, 1, -1) == 0
    phi = np.zeros((32, 6))
    n = [np.zeros(ens.n_nodes) for _ in range(2)]
    L.bt_eval(T, X.ctypes.data, G.ctypes.data, 32, 12, phi.ctypes.data, n[0].ctypes.data, n[1].ctypes.data)
    L.bt_free(T)
    # path by path: merged intervals, [lo, hi)
    ref = np.zeros((32, 6))
    x, w = np.polynomial.legendre.leggauss(12)
    t, w = 0.5 * (x + 1), 0.5 * w
    for k in range(ens.n_trees):
        b = int(ens.node_offsets[k])
        stack = [(0, {})]
        while stack:
            v, el = stack.pop()
            g = b + v
            if ens.left[g] >= 0:
                f, thr = int(ens.feature[g]), ens.threshold[g]
                for c, left in ((int(ens.left[g]), True), (int(ens.right[g]), False)):
                    z, lo, hi = el.get(f, (1.0, -np.inf, np.inf))
                    e = dict(el)
                    e[f] = (z * float(ens.z[b + c]), lo if left else max(lo, thr), min(hi, thr) if left else hi)
                    stack.append((c, e))
                continue
            fs = sorted(el)
            z = np.array([el[f][0] for f in fs])
            o = np.stack([(X[:, f] >= el[f][1]) & (X[:, f] < el[f][2]) for f in fs], 1).astype(float)
            a = z[:, None] + t * (o - z)[:, :, None]
            for i, f in enumerate(fs):
                rest = np.prod(np.delete(a, i, 1), 1)
                ref[:, f] += float(ens.leaf_value[g]) * (o - z)[:, i] * (rest * w).sum(1)
    assert np.abs(phi - ref).max() <= 1e-11 * np.abs(ref).max()


def test_blocks_of_every_height_and_a_leaf_in_one_block_each(host_lib):
    L = load(host_lib)
    ens = tiny_ensemble(21, n_trees=4, depth=8, F=10, n_train=800)
    T = tables(L, ens)
    assert L.bt_build(T, 0, -1) == 0
    assert all(L.bt_blocks(T, h) > 0 for h in range(4))
    L.bt_free(T)


OUT_OF_MEMORY = """
import sys
sys.path[:0] = [{root!r}, {tests!r}]
import synth
import test_block_tables as t
L = t.load({lib!r})
ens = synth.grow(30, 16, 12, 20, 60000, 1.0, min_rows=2)  # many threads' worth of nodes
T = t.tables(L, ens)
for n in (0, 1, 5, 20, 100):
    for call in (lambda: L.bt_build(T, 1, n), lambda: L.bt_prepare(T, n)):
        assert call() == 1, n
assert L.bt_build(T, 1, -1) == 0 and L.bt_prepare(T, -1) == 0
print("ok", ens.n_nodes)
"""


def test_out_of_memory_is_an_error_on_every_thread(host_lib):
    code = OUT_OF_MEMORY.format(root=ROOT, tests=os.path.join(ROOT, "tests"), lib=host_lib)
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.startswith("ok"), (r.returncode, r.stderr[-500:])
