"""The pixel-driven back projector at pitches about and below one pixel with
scans about a diagonal, where a pixel step stays below one bin although a tile
reaches over more bins than at a pitch of one (one pixel at a time, or 2 x 2
blocks where their window still holds the tile)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# positions off by at most 4 ulp(32) / 2 ~ 8e-6 bins, sums by a few 2^-24: the projectors' parity bound
TOL = 1e-5

GEOMS = [
    # N, n_angles, n_det, start, range, det_spacing
    (128, 60, 256, 40, 10, 0.8),
    (128, 12, 256, 42, 6, 0.75),
    (128, 30, 220, 30, 30, 0.9),
    (256, 4, 512, 45, 360, 0.71),
    (64, 4, 100, 45, 360, 0.75),
    (64, 60, 100, 35, 20, 0.9),
    (65, 33, 131, 131, 8, 0.72),
    (64, 4, 100, 45, 360, 0.94),       # blocks, at the edge of their window
    (64, 20, 100, 43, 4, 0.95),
    (131, 12, 200, 223, 4, 0.96),
    (700, 16, 1300, 38, 14, 0.8),      # as large as takes 64-row tiles
    (700, 130, 1060, 43, 4, 0.96),
    (1024, 8, 1600, 45, 360, 0.97),
]


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2110_01481_gb300 as P
    return P


@pytest.mark.parametrize("geom", GEOMS)
def test_back_parity_about_the_diagonals(P, oracle_mod, geom):
    import torch
    g, og = P.Geometry(*geom), oracle_mod.Geometry(*geom)
    b = np.random.default_rng(15).standard_normal(g.m).astype(np.float32)
    out = torch.full((g.n,), float("nan"), device="cuda")
    got = P.backproject(g, torch.tensor(b, device="cuda"), out=out).double().cpu().numpy()
    ref = oracle_mod.backproject(og, b.astype(np.float64))
    assert np.linalg.norm(got - ref) <= TOL * np.linalg.norm(ref)
    assert np.abs(got - ref).max() <= 10 * TOL * np.abs(ref).max()
