"""The Givens update and y_k inside the one-launch CGS2 step, against FP64 least
squares on the step's own Hessenberg matrix: every k where the column (32
entries per lane slot, four at a time in the recurrence) or y_k (two slots)
starts a new part."""
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


def _least_squares(H, k, beta):
    e = np.zeros(k + 1)
    e[0] = beta
    y = np.linalg.lstsq(H[:k + 1, :k], e, rcond=None)[0]
    return y, np.linalg.norm(e - H[:k + 1, :k] @ y)


def _noise(P, seed):
    import torch
    g = P.Geometry(64, 90, 91)
    torch.manual_seed(seed)
    return g, torch.randn(g.m, device="cuda")


def test_rotated_column_up_to_the_largest_step(P):
    g, b = _noise(P, 1)
    K = 128
    r = P.ab_gmres(g, b, K, keep_workspace=True)
    assert r.iters == K
    H = r.hessenberg(g, "ab", K).cpu().numpy()
    beta = r.history[0]
    for k in (1, 2, 5, 31, 32, 33, 34, 64, 65, 97, 127, 128):
        # both are FP64 on one matrix: k rotations of a few roundings each
        assert abs(r.history[k] - _least_squares(H, k, beta)[1]) <= 1e-10 * beta, k


def test_iterate_of_every_step(P):
    """BA with a target that is never met: x_k = W_k y_k is formed in each step,
    and the history is its residual."""
    import torch
    g, b = _noise(P, 2)
    K = 64
    r = P.ba_gmres(g, b, K, keep_workspace=True, noise_norm=1e-9)
    assert r.iters == K
    H = r.hessenberg(g, "ba", K).cpu().numpy()
    W = r.basis(g, "ba", K).double()
    beta = float(P.backproject(g, b).double().norm())
    nb = float(b.double().norm())
    for k in (1, 2, 31, 32, 33, 34, 63, 64):
        y, _ = _least_squares(H, k, beta)
        x = (W[:k].T @ torch.tensor(y, device="cuda")).float()
        res = float((b.double() - P.project(g, x).double()).norm())
        # FP32 x_k and A x_k on either side: k + 16 roundings of ||x_k|| entries
        assert abs(r.history[k] - res) <= (k + 16) * 2.0 ** -23 * nb, k
