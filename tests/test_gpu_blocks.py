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
