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
