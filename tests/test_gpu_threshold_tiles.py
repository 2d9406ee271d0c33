"""B_tau at the edges of its tiles (one tile, a middle row shared by a pixel and
its reflection, several ragged tiles): between the oracle's B_tau without and
with the entries that lie within rounding of the threshold."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2110_01481_gb300 as P
    return P


@pytest.mark.parametrize("tau", [0.1, 0.45])
@pytest.mark.parametrize("N", [31, 32, 33, 70])
def test_thresholded_tiles(P, oracle_mod, N, tau):
    import scipy.sparse as sp
    import torch
    args = (N, 21, N + 9, 0, 360, 1.0)
    g, og = P.Geometry(*args, back_model="threshold", back_tau=tau), oracle_mod.Geometry(*args)
    A = oracle_mod.matrix_A(og).tocoo()
    amax = A.data.max()
    # the GPU decides in FP32: positions off by at most 8e-6 bins, weights of slope sqrt(2)
    eps = 2e-5 * amax
    B = [sp.csr_matrix((A.data[keep], (A.col[keep], A.row[keep])), shape=(og.n, og.m))
         for keep in (A.data >= tau * amax + eps, A.data >= tau * amax - eps)]
    b = np.random.default_rng(17).uniform(0.5, 1.0, og.m).astype(np.float32)      # b > 0: monotone in the kept set
    low, high = (M @ b.astype(np.float64) for M in B)
    out = torch.full((g.n,), float("nan"), device="cuda")
    got = P.backproject(g, torch.tensor(b, device="cuda"), out=out).double().cpu().numpy()
    tol = 2e-5 * high.max()
    assert (got >= low - tol).all() and (got <= high + tol).all()
    # few entries are that close to the threshold, so this is no slack: nearly all pixels are pinned
    assert np.count_nonzero(high - low > tol) <= 0.2 * og.n
