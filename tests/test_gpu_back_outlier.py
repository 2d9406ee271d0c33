"""A large detector bin reaches only the pixels that interpolate it: with one
impulse the others are exactly zero, and with one outlier in unit noise they are
what the noise alone gives, in every form of the pixel-driven back projector."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

GEOMS = [
    # N, n_angles, n_det, start, range, det_spacing
    (64, 90, 91, 0, 180, 1.0),         # blocks; half-integer positions along the axes
    (65, 92, 93, 0, 360, 1.0),         # whole positions along the axes: weights of exactly zero and one
    (700, 20, 990, 0, 180, 1.0),       # 64-row tiles
    (64, 52, 60, 0, 180, 1.5),         # the far corner may take its block's lowest bin
    (63, 24, 31, 0, 360, 2.0),
    (64, 20, 100, 43, 4, 0.95),        # a pitch below one that takes blocks
    (47, 30, 71, 0, 180, 0.8),         # one pixel at a time
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


def _untouched(geom, a, d):
    """Pixels at least a bin (and a margin for the rounding of positions) from bin d of angle a."""
    N, n_angles, n_det, start, range_, ds = geom
    th = np.deg2rad(start + a * range_ / n_angles)
    t = np.arange(N) - 0.5 * (N - 1)
    u = (t[None, :] * np.cos(th) + t[:, None] * np.sin(th)) / ds + 0.5 * (n_det - 1)
    dist = np.abs(u - d)
    exact = np.abs(dist - 1.0) < 1e-9          # on an axis with whole positions: the weight is zero
    return ((dist >= 1.0 + 1e-4) | (exact & (a * range_ % (90 * n_angles) == 0) & (start % 90 == 0))).ravel()


@pytest.mark.parametrize("geom", GEOMS)
def test_an_outlier_stays_with_its_pixels(P, oracle_mod, geom):
    import torch
    N, n_angles, n_det = geom[:3]
    g, og = P.Geometry(*geom), oracle_mod.Geometry(*geom)
    noise = np.random.default_rng(16).standard_normal((n_angles, n_det)).astype(np.float32)
    ref = oracle_mod.backproject(og, noise.astype(np.float64).ravel()).ravel()
    # positions off by at most 8e-6 bins and sums by a few 2^-24, as in the parity tests of the largest entry
    bound = 1e-4 * np.abs(ref).max()
    for a, d in ((0, n_det // 2), (0, n_det // 2 + 4), (n_angles // 6, n_det // 2 - 3), (n_angles // 4, n_det // 2 + 5),
                 (n_angles // 2, n_det // 2), (n_angles - 1, n_det // 3)):
        free = _untouched(geom, a, d)
        one = np.zeros((n_angles, n_det), np.float32)
        one[a, d] = 1.0
        got = P.backproject(g, torch.tensor(one.ravel(), device="cuda")).cpu().numpy()
        assert np.count_nonzero(got[free]) == 0, (a, d)
        assert np.count_nonzero(got) > 0
        b = noise.copy()
        b[a, d] = 1e6
        got = P.backproject(g, torch.tensor(b.ravel(), device="cuda")).double().cpu().numpy()
        assert np.abs(got - ref)[free].max() <= bound, (a, d)
