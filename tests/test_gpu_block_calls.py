"""Calls around the block tables: what a call may rely on besides its inputs
(captures, workspaces, saved tuning files) and inputs at the edge of what the
kernels' FP32 sums hold, against the oracle."""
import numpy as np
import pytest

import oracle
import synth
from helpers import rel_err_rows

pytestmark = pytest.mark.gpu

TOL32 = 1e-5  # FP32 tables: the bound every FP32 test of this suite uses


@pytest.fixture(scope="module")
def qts():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_04497_gb300 import build as b

    b.build()
    import paper_2605_04497_gb300 as q

    return q


def _rel(a, b):
    return np.abs(a - b).max() / max(np.abs(b).max(), 1e-300)


def _request(qts, E, X, G=None):
    """One batched request on new outputs; without G forward only."""
    import torch

    new = lambda *s: torch.empty(s, dtype=torch.float64, device="cuda")
    it = dict(ens=E, X=X, phi=new(len(X), E.n_features + 1))
    if G is not None:
        it.update(grad_phi=G, d_leaf=new(E.n_nodes), d_z=new(E.n_nodes))
    return it


@pytest.mark.parametrize("F", [9, 130])  # two samples per lane, one sample per lane
def test_bias_weights_stay_out_of_the_leaf_gradients(qts, F):
    """grad_phi's last column weighs E[f]; where its sum cancels, whatever its
    size, it leaves the leaf gradients' digits alone, at leaves of every height."""
    import torch

    ens = synth.grow(9500, 6, 6, F, 2000, 0.5, min_rows=3)
    M = 64
    X = synth.normal(9500, synth.STREAM_X, (M, F))
    G = synth.normal(9500, synth.STREAM_GRAD, (M, F + 1))
    G[:, F] = np.where(np.arange(M) % 2, 1e4, -1e4)  # their sum is exactly zero
    dl_ref, dz_ref = oracle.grad_exact(ens, X, G)
    E = qts.Ensemble.from_arrays(ens)
    Xd, Gd = torch.from_numpy(X).cuda(), torch.from_numpy(G).cuda()
    dl, dz = qts.shap_backward(E, Xd, Gd)
    it = _request(qts, E, Xd, Gd)
    qts.batched_fwd_bwd(qts.make_requests([it]))
    E.sync_status()
    for a, b in ((dl, dl_ref), (dz, dz_ref), (it["d_leaf"], dl_ref), (it["d_z"], dz_ref)):
        assert _rel(a.cpu().numpy(), b) <= TOL32
    E.close()


@pytest.mark.parametrize("kind", ["adjoint", "pairs"])
def test_captured_call_survives_a_larger_one(qts, kind):
    """A graph that holds the workspace is replayed after an adjoint call of more
    samples, which needs a larger one: the captured one must not have been freed."""
    import torch

    F, M, M2 = 10, 400000, 2000000
    ens = synth.grow(9600, 2, 4, F, 2000, 0.5, min_rows=3)
    E = qts.Ensemble.from_arrays(ens)
    X = torch.from_numpy(synth.normal(9600, synth.STREAM_X, (M2, F))).cuda()
    G = torch.from_numpy(synth.normal(9600, synth.STREAM_GRAD, (M2, F + 1))).cuda()
    new = lambda: torch.zeros(E.n_nodes, dtype=torch.float64, device="cuda")
    outs, out2 = (new(), new()), (new(), new())
    rows = M if kind == "adjoint" else 100000
    Xs, Gs = X[:rows].contiguous(), G[:rows].contiguous()
    if kind == "pairs":
        outs = (torch.zeros((rows, F + 1, F + 1), dtype=torch.float32, device="cuda"),)

    def call():
        if kind == "adjoint":
            qts.shap_backward(E, Xs, Gs, d_leaf=outs[0], d_z=outs[1])
        else:
            qts.shap_interactions(E, Xs, out=outs[0])

    call()
    torch.cuda.synchronize()
    ref = [o.cpu().numpy() for o in outs]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    qts.shap_backward(E, X, G, d_leaf=out2[0], d_z=out2[1])
    torch.cuda.synchronize()
    # transposed copies of the M2 samples; the captured workspace is not given back
    grown = 2 * 4 * (F + 1) * M2
    assert free - torch.cuda.mem_get_info()[0] >= 0.95 * grown
    for o in outs:
        o.zero_()
    g.replay()
    torch.cuda.synchronize()
    for o, r in zip(outs, ref):
        assert _rel(o.cpu().numpy(), r) <= (1e-9 if kind == "adjoint" else 1e-6)
    E.sync_status()
    E.close()


@pytest.mark.parametrize("kind", ["fp64", "fp32", "few", "adjoint", "adjoint-after-forward"])
def test_first_call_under_capture(qts, kind):
    """The tables that a call builds on first use may be built under capture (the
    FP64 forward, and the adjoint's part after a forward)."""
    import torch

    F, M = 7, 5 if kind == "few" else 40
    ens = synth.grow(9700, 4, 5, F, 2000, 0.5, min_rows=3)
    Xh = synth.normal(9700, synth.STREAM_X, (M, F))
    Gh = synth.normal(9700, synth.STREAM_GRAD, (M, F + 1))
    X, G = torch.from_numpy(Xh).cuda(), torch.from_numpy(Gh).cuda()
    E = qts.Ensemble.from_arrays(ens, fp64=kind == "fp64")
    if kind == "adjoint-after-forward":
        qts.shap_values(E, X)
    phi = torch.zeros((M, F + 1), dtype=torch.float64, device="cuda")
    dl = torch.zeros(E.n_nodes, dtype=torch.float64, device="cuda")
    dz = torch.zeros_like(dl)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        if kind.startswith("adjoint"):
            qts.shap_backward(E, X, G, d_leaf=dl, d_z=dz)
        else:
            qts.shap_values(E, X, out=phi)
    g.replay()
    E.sync_status()
    if kind.startswith("adjoint"):
        for a, b in zip((dl, dz), oracle.grad_exact(ens, Xh, Gh)):
            assert _rel(a.cpu().numpy(), b) <= TOL32
    else:
        assert rel_err_rows(phi.cpu().numpy(), oracle.shap_exact(ens, Xh)).max() <= TOL32
    E.close()


@pytest.mark.parametrize("M", [1, 8192, 8193, 20000])  # a thread block sums 8,192 samples' weights
def test_weights_of_the_expected_value(qts, M):
    """The gradient through E[f] alone: the sum of grad_phi's last column over all
    samples, times a constant per node.  FP32 weights, FP64 sums."""
    import torch

    ens = synth.grow(9800, 3, 3, 4, 2000, 0.5, min_rows=3)
    E = qts.Ensemble.from_arrays(ens)
    X = torch.from_numpy(synth.normal(9800, synth.STREAM_X, (M, 4))).cuda()
    g = synth.normal(9800, synth.STREAM_GRAD, (M,)) + np.float32(0.5)
    G = torch.zeros((M, 5), device="cuda")
    G[:, 4] = torch.from_numpy(g).cuda()
    one = np.zeros((1, 5), np.float32)
    one[0, 4] = 1.0
    total = g.astype(np.float64).sum()
    ref = [total * r for r in oracle.grad_exact(ens, np.zeros((1, 4), np.float32), one)]
    dl, dz = qts.shap_backward(E, X, G)
    it = _request(qts, E, X, G)
    for _ in range(2):  # the sum starts at zero in a replay too
        qts.batched_fwd_bwd(qts.make_requests([it]))
    E.sync_status()
    # other gradients are zero, so only the FP64 sum's order differs
    for a, b in zip((dl, dz, it["d_leaf"], it["d_z"]), ref + ref):
        assert _rel(a.cpu().numpy(), b) <= 1e-12
    E.close()


def test_adjoint_in_slabs_of_samples(qts):
    """More samples than the transposed copies hold at a time (41,728 at F = 800):
    the workspace stays bounded, and the gradients are the sum over two halves."""
    import torch

    F, M, cut = 800, 90001, 16384
    ens = synth.grow(9900, 2, 4, F, 2000, 0.5, min_rows=3)
    E = qts.Ensemble.from_arrays(ens)
    gen = torch.Generator("cuda").manual_seed(9900)
    X = torch.randn((M, F), device="cuda", generator=gen)
    G = torch.randn((M, F + 1), device="cuda", generator=gen)
    new = lambda: torch.empty(E.n_nodes, dtype=torch.float64, device="cuda")
    dl, dz = new(), new()
    a = qts.shap_backward(E, X[:cut], G[:cut])
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    qts.shap_backward(E, X, G, d_leaf=dl, d_z=dz)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] <= 280 << 20  # all samples at once: 577 MB
    b = qts.shap_backward(E, X[cut:].contiguous(), G[cut:].contiguous())
    E.sync_status()
    # the cut and the slabs lie on whole tiles of samples, so only the order of FP64 sums differs
    for got, p, q in ((dl, a[0], b[0]), (dz, a[1], b[1])):
        assert _rel(got.cpu().numpy(), (p + q).cpu().numpy()) <= 1e-11
    E.close()


@pytest.mark.parametrize("T,depth,F,M", [(1, 1, 1, 20000), (1, 2, 3, 19999), (3, 6, 12, 20001), (1, 10, 40, 40033),
                                         (2, 14, 9, 40000), (0, 41, 50, 40031)])
@pytest.mark.parametrize("missing", [False, True])
def test_small_ensemble_many_samples(qts, T, depth, F, M, missing):
    """A warp walks all blocks for its samples (every class of widths, whole and
    ragged tiles, clean tiles beside tiles with NaN and +inf); 0 trees: a chain."""
    import torch

    from helpers import caterpillar_ensemble

    ens = (synth.grow(9850 + depth, T, depth, F, 3000, 0.5, min_rows=3) if T else
           caterpillar_ensemble(9850, [depth, 20, 9], F))
    X = synth.normal(9850 + depth, synth.STREAM_X, (M, F))
    r = np.random.default_rng(9850)
    rows = np.unique(np.concatenate([np.arange(40), M - 1 - np.arange(40), r.integers(0, M, 60)]))
    if missing:
        X[::3][r.random(X[::3].shape) < 0.2] = np.nan
        X[64:96] = np.abs(X[64:96])
    ref = oracle.shap_exact(ens, np.ascontiguousarray(X[rows]))
    E = qts.Ensemble.from_arrays(ens)
    Xd = torch.from_numpy(X).cuda()
    few = qts.shap_values(E, Xd[:16], qts.EXACT_NODES)  # another kernel
    for n_quad in (qts.EXACT_NODES,) + ((8, 11) if T else (21,)):
        phi = qts.shap_values(E, Xd, n_quad)
        E.sync_status()
        assert rel_err_rows(phi[torch.from_numpy(rows).cuda()].cpu().numpy(), ref).max() <= TOL32, n_quad
        assert rel_err_rows(phi[:16].cpu().numpy(), few.cpu().numpy()).max() <= TOL32
    E.close()


# (trees, 0: a chain, its depth, F, M): pairs without a tile in shared memory (F = 60, at a
# mean width on either side of the one-row line) and with one, wide and padded widths,
# few and many samples
PAIR_ROUTES = [(4, 5, 60, 1), (4, 5, 60, 40), (2, 17, 60, 1), (2, 17, 60, 33), (2, 12, 24, 4), (2, 12, 24, 5),
               (2, 12, 24, 40), (0, 30, 40, 5), (0, 30, 40, 40), (1, 4, 10, 16), (1, 4, 10, 17), (3, 7, 48, 40), (0, 30, 60, 5), (0, 30, 60, 40)]


@pytest.mark.parametrize("T,depth,F,M", PAIR_ROUTES)
@pytest.mark.parametrize("kind", ["clean", "missing", "categories"])
def test_pairs_on_either_tables(qts, T, depth, F, M, kind):
    import torch

    from helpers import caterpillar_ensemble

    ens = (synth.grow(9950 + depth, T, depth, F, 600, 0.5, min_rows=3) if T else
           caterpillar_ensemble(9950, [depth, 18, 4], F))
    X = synth.normal(9950 + depth, synth.STREAM_X, (M, F))
    if kind == "categories":
        cats = list(range(0, F, 3))
        ens = synth.make_categorical(ens, cats, 6, 9951)
        X = synth.categorical_columns(X, cats, 6, 9952)
    elif kind == "missing":
        X[np.random.default_rng(9950).random(X.shape) < 0.2] = np.nan
    E = qts.Ensemble.from_arrays(ens)
    sii, phi = oracle.sii_exact(ens, X)
    ref = oracle.interaction_matrix(sii, phi)
    scale = np.maximum(np.abs(phi.sum(1)), np.abs(phi[:, :-1]).max(1))
    for n_quad in (qts.EXACT_NODES, 16, 17):  # 17: an odd rule
        got = qts.shap_interactions(E, torch.from_numpy(X).cuda(), n_quad).cpu().numpy().astype(np.float64)
        E.sync_status()
        assert (np.abs(got - ref).reshape(M, -1).max(1) / scale).max() <= TOL32, n_quad
    E.close()


def test_large_forward_only_requests_in_a_batch(qts):
    """Forward-only requests that fill the chip run the forward's own kernels inside the
    batch's graph, beside small ones and one with gradients; replays start from
    new inputs."""
    import torch

    sizes = [(60, 8, 20, 3000), (5, 4, 6, 40), (30, 13, 130, 1500), (20, 6, 12, 200)]
    items, hosts = [], []
    for i, (T, depth, F, M) in enumerate(sizes):
        ens = synth.grow(9960 + i, T, depth, F, 5000, 0.5, min_rows=3)
        X = synth.normal(9960 + i, synth.STREAM_X, (M, F))
        X[::7, 0] = np.nan
        G = torch.from_numpy(synth.normal(9960, synth.STREAM_GRAD, (M, F + 1))).cuda() if i == 3 else None
        items.append(_request(qts, qts.Ensemble.from_arrays(ens), torch.from_numpy(X).cuda(), G))
        hosts.append(ens)
    reqs = qts.make_requests(items)
    rows = np.arange(0, 40)
    for n_quad in (8, qts.EXACT_NODES):
        for _ in range(2):
            qts.batched_fwd_bwd(reqs, n_quad)
            assert qts.batched_kernel_count() > 4
            for ens, it in zip(hosts, items):
                it["ens"].sync_status()
                ref = oracle.shap_exact(ens, it["X"].cpu().numpy()[rows])
                assert rel_err_rows(it["phi"][:40].cpu().numpy(), ref).max() <= TOL32
                last = qts.shap_values(it["ens"], it["X"][-16:].contiguous(), n_quad)
                assert rel_err_rows(it["phi"][-16:].cpu().numpy(), last.cpu().numpy()).max() <= TOL32
                it["X"].mul_(-1.0)
    assert qts.batched_autotune(reqs, 8, max_samples=0)
    qts.batched_fwd_bwd(reqs)
    for ens, it in zip(hosts, items):
        ref = oracle.shap_exact(ens, it["X"].cpu().numpy()[rows])
        assert rel_err_rows(it["phi"][:40].cpu().numpy(), ref).max() <= TOL32
        it["ens"].close()


def test_tuning_cache_of_an_earlier_format(qts, tmp_path):
    """Entries of another meaning are kept in the file and not used; a fitting entry is
    taken only with a value that the tuner writes."""
    import json
    import math

    import torch

    ens = synth.grow(9970, 12, 5, 9, 2000, 0.5, min_rows=3)
    E = qts.Ensemble.from_arrays(ens)
    Xh = synth.normal(9970, synth.STREAM_X, (300, 9))
    X = torch.from_numpy(Xh).cuda()
    path = tmp_path / "tune.json"
    old = {f"{D}|{int(math.log2(9))}|{int(math.log2(300))}": [8, 2048, 32, 8, 2147483647, 0]
           for D, _ in E.info()["buckets"]}
    path.write_text(json.dumps(old))
    qts.autotune(E, X, str(path))
    data = json.loads(path.read_text())
    new = {k: v for k, v in data.items() if k not in old}
    assert {k: v for k, v in data.items() if k in old} == old
    assert len(new) == len(old) and all(v in ([0], [128], [256], [512], [1024], [2048]) for v in new.values())
    # a spoiled entry under the current key is timed anew
    path.write_text(json.dumps({k: [2147483647] for k in new}))
    qts.autotune(E, X, str(path))
    assert all(v[0] <= 2048 for v in json.loads(path.read_text()).values())
    phi = qts.shap_values(E, X)
    E.sync_status()
    assert rel_err_rows(phi.cpu().numpy(), oracle.shap_exact(ens, Xh)).max() <= TOL32
    E.close()
