"""Block tables (small subtrees evaluated against the elements their leaves
share): the sizes where a block's shape, a sample tile or a launch class ends,
against the oracle."""
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


# (trees, depth, F, M, full): whole trees in one block of height 1, 2, 3 (no
# shared element); one level more; two features only (every split below the
# second repeats one, so blocks are cut at each node); repeats and new features
# mixed; one class of widths after the other; a phi tile per warp no longer
# fits (F = 300); sample tiles of 32 with a remainder of 1, 31 and none
SHAPES = [
    (3, 1, 4, 17, True), (3, 2, 6, 31, True), (3, 3, 9, 32, True), (2, 4, 9, 33, True),
    (3, 9, 2, 64, False), (4, 8, 5, 65, False), (6, 8, 40, 127, False), (3, 13, 20, 96, False),
    (2, 17, 60, 40, False), (3, 6, 300, 50, False),
]


@pytest.mark.parametrize("T,depth,F,M,full", SHAPES)
@pytest.mark.parametrize("missing", [False, True])
def test_forward_shapes(qts, T, depth, F, M, full, missing):
    import torch

    ens = synth.grow(9000 + depth, T, depth, F, 4000, 0.5, min_rows=3, full_depth=full)
    X = synth.normal(9000 + depth, synth.STREAM_X, (M, F))
    if missing:
        X[np.random.default_rng(depth).random(X.shape) < 0.2] = np.nan
    E = qts.Ensemble.from_arrays(ens)
    ref = oracle.shap_exact(ens, X)
    for n_quad in (8, qts.EXACT_NODES, 11):  # 11: an odd rule, padded to node pairs
        phi = qts.shap_values(E, torch.from_numpy(X).cuda(), n_quad).cpu().numpy()
        E.sync_status()
        assert rel_err_rows(phi, ref).max() <= TOL32, n_quad
    E.close()


def _rel(a, b):
    return np.abs(a - b).max() / max(np.abs(b).max(), 1e-300)


@pytest.mark.parametrize("T,depth,F,M,full", SHAPES)
@pytest.mark.parametrize("missing", [False, True])
def test_adjoint_and_batched_shapes(qts, T, depth, F, M, full, missing):
    """The fused pass and the plain adjoint on the same shapes (F = 300: one
    sample per lane and a shared phi tile)."""
    import torch

    ens = synth.grow(9100 + depth, T, depth, F, 4000, 0.5, min_rows=3, full_depth=full)
    X = synth.normal(9100 + depth, synth.STREAM_X, (M, F))
    G = synth.normal(9100 + depth, synth.STREAM_GRAD, (M, F + 1))
    if missing:
        X[np.random.default_rng(depth).random(X.shape) < 0.2] = np.nan
    E = qts.Ensemble.from_arrays(ens)
    Xd, Gd = torch.from_numpy(X).cuda(), torch.from_numpy(G).cuda()
    ref = oracle.shap_exact(ens, X)
    dl_ref, dz_ref = oracle.grad_exact(ens, X, G)
    new = lambda *s: torch.empty(s, dtype=torch.float64, device="cuda")
    for n_quad in (8, qts.EXACT_NODES, 11):
        dl, dz = qts.shap_backward(E, Xd, Gd, n_quad)
        it = dict(ens=E, X=Xd, grad_phi=Gd, phi=new(M, F + 1), d_leaf=new(E.n_nodes), d_z=new(E.n_nodes))
        qts.batched_fwd_bwd(qts.make_requests([it]), n_quad)
        E.sync_status()
        assert rel_err_rows(it["phi"].cpu().numpy(), ref).max() <= TOL32, n_quad
        for a, b in ((dl, it["d_leaf"]), (dz, it["d_z"])):
            r = dl_ref if a is dl else dz_ref
            assert _rel(a.cpu().numpy(), r) <= TOL32 and _rel(b.cpu().numpy(), r) <= TOL32, n_quad
        # forward only
        it = dict(ens=E, X=Xd, phi=new(M, F + 1))
        qts.batched_fwd_bwd(qts.make_requests([it]), n_quad)
        assert rel_err_rows(it["phi"].cpu().numpy(), ref).max() <= TOL32, n_quad
    E.close()


@pytest.mark.parametrize("T,depth,F,M,full", [s for s in SHAPES if s[0] * s[1] < 40])
@pytest.mark.parametrize("rows", [None, 1, 5])
def test_interaction_shapes(qts, T, depth, F, M, full, rows):
    """Pairs between shared elements, elements and nodes, and nodes above nodes;
    F = 300: the pair tile does not fit; few rows: lanes hold different blocks."""
    import torch

    ens = synth.grow(9200 + depth, T, depth, F, 1500, 0.5, min_rows=3, full_depth=full)
    X = synth.normal(9200 + depth, synth.STREAM_X, (rows or min(M, 40), F))
    X[-1, :2] = np.nan
    E = qts.Ensemble.from_arrays(ens)
    sii, phi = oracle.sii_exact(ens, X)
    ref = oracle.interaction_matrix(sii, phi)
    scale = np.maximum(np.abs(phi.sum(1)), np.abs(phi[:, :-1]).max(1))
    for n_quad in (8, qts.EXACT_NODES, 11):
        got = qts.shap_interactions(E, torch.from_numpy(X).cuda(), n_quad).cpu().numpy().astype(np.float64)
        E.sync_status()
        assert (np.abs(got - ref).reshape(len(X), -1).max(1) / scale).max() <= TOL32, n_quad
    E.close()


@pytest.mark.parametrize("M", [3, 40])
def test_infinite_inputs_as_on_the_path_tables(qts, M):
    """Infinities take the sides that the path tables' half-open intervals give
    them: the allocation-free interactions run on those tables, and their rows
    sum to phi."""
    import torch

    ens = synth.grow(9300, 8, 7, 7, 3000, 0.5, min_rows=3)
    X = synth.normal(9300, synth.STREAM_X, (M, 7))
    r = np.random.default_rng(3).random(X.shape)
    X[r < 0.15], X[(r >= 0.15) & (r < 0.3)] = np.inf, -np.inf
    E, E64 = qts.Ensemble.from_arrays(ens), qts.Ensemble.from_arrays(ens, fp64=True)
    Xd = torch.from_numpy(X).cuda()
    ref = qts.shap_interactions_noalloc(E, Xd, torch.empty((M, 8, 8), dtype=torch.float32, device="cuda"))
    ref = ref.cpu().numpy().astype(np.float64)
    scale = np.abs(ref).max()
    assert np.isfinite(ref).all()
    for e in (E, E64):
        phi = qts.shap_values(e, Xd).cpu().numpy()
        assert np.abs(phi[:, :7] - ref[:, :7, :7].sum(2)).max() <= TOL32 * scale
    got = qts.shap_interactions(E, Xd).cpu().numpy()
    assert np.abs(got - ref).max() <= TOL32 * scale
    it = dict(ens=E, X=Xd, grad_phi=torch.ones((M, 8), device="cuda"),
              phi=torch.empty((M, 8), dtype=torch.float64, device="cuda"),
              d_leaf=torch.empty(E.n_nodes, dtype=torch.float64, device="cuda"),
              d_z=torch.empty(E.n_nodes, dtype=torch.float64, device="cuda"))
    qts.batched_fwd_bwd(qts.make_requests([it]))
    assert np.abs(it["phi"].cpu().numpy()[:, :7] - ref[:, :7, :7].sum(2)).max() <= TOL32 * scale
    E.close()
    E64.close()


def test_captured_adjoint_of_more_samples(qts):
    """A capture may hold an adjoint call that needs more workspace than any call
    before it."""
    import torch

    ens = synth.grow(9400, 5, 6, 9, 2000, 0.5, min_rows=3)
    E = qts.Ensemble.from_arrays(ens)
    M = 60000
    X = torch.from_numpy(synth.normal(9400, synth.STREAM_X, (M, 9))).cuda()
    G = torch.from_numpy(synth.normal(9400, synth.STREAM_GRAD, (M, 10))).cuda()
    qts.shap_backward(E, X[:20].contiguous(), G[:20].contiguous())
    dl = torch.zeros(E.n_nodes, dtype=torch.float64, device="cuda")
    dz = torch.zeros_like(dl)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        qts.shap_backward(E, X, G, d_leaf=dl, d_z=dz)
    g.replay()
    torch.cuda.synchronize()
    dl2, dz2 = qts.shap_backward(E, X, G)
    assert _rel(dl.cpu().numpy(), dl2.cpu().numpy()) <= 1e-9
    assert _rel(dz.cpu().numpy(), dz2.cpu().numpy()) <= 1e-9
    E.close()
