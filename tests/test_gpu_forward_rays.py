"""The forward projector's walks: rays that miss the image, which must come out
zero whatever their neighbours in the warp do (a detector much wider than the
image, ragged last groups of rays, image sides that are no multiple of 4)."""
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


@pytest.mark.parametrize("N,Na,Nd,start,rng", [
    (30, 24, 301, 0, 180),      # 13 rays in the last group, 135 bins off the image at 0 degrees
    (29, 9, 403, 45, 360),
    (13, 40, 200, 0, 180),      # a group of rays wider than the image
    (66, 90, 333, 0, 180),
    (999, 36, 1413, 0, 180),    # the ordinary detector of a large odd image
])
def test_rays_off_the_image_are_zero(P, oracle_mod, N, Na, Nd, start, rng):
    import torch
    g, og = P.Geometry(N, Na, Nd, start, rng), oracle_mod.Geometry(N, Na, Nd, start, rng)
    x = np.random.default_rng(9).uniform(0.5, 1.0, (N, N)).astype(np.float32)
    ref = oracle_mod.forward(og, x.astype(np.float64))
    ctx = P.Context.get(torch.device("cuda", 0))
    xt = torch.tensor(x.ravel(), device="cuda")
    try:
        for angles, per_warp in ((0, 1), (8, 1), (4, 1), (8, 4), (16, 4)):
            ctx.set_tiles(angles, 32 if angles else 0, per_warp)
            got = P.project(g, xt).double().cpu().numpy()
            assert np.count_nonzero(got[ref == 0.0]) == 0, (angles, per_warp)
            assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)
    finally:
        ctx.set_tiles(0, 0)
