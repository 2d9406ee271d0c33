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


# N, n_angles, n_det, start, range, det_spacing: the drive changes inside a
# group of four or eight angles (at 45 and 135 degrees, odd counts), groups of
# one (widely spaced angles), negative cosines, a last group with one angle,
# clamped walks (very coarse pitch), one angle alone
GROUPS = [(40, 1, 57, 30, 180, 1.0), (40, 3, 57, 0, 180, 1.0), (50, 9, 71, 0, 360, 1.0), (64, 61, 91, 40, 10, 1.0),
          (64, 90, 91, 0, 180, 1.0), (61, 121, 87, -50, 180, 1.0), (90, 200, 128, 100, 360, 1.0), (48, 33, 90, 0, 180, 0.75),
          (40, 37, 12, 0, 180, 7.0), (150, 16, 213, 130, 10, 1.0)]


@pytest.mark.parametrize("geom", GROUPS)
def test_angle_groups_of_every_shape(P, oracle_mod, geom):
    import torch
    g, og = P.Geometry(*geom), oracle_mod.Geometry(*geom)
    x = np.random.default_rng(12).standard_normal((g.N, g.N)).astype(np.float32)
    ref = oracle_mod.forward(og, x.astype(np.float64))
    ctx = P.Context.get(torch.device("cuda", 0))
    xt = torch.tensor(x.ravel(), device="cuda")
    outs = []
    try:
        for angles, per_warp in ((0, 1), (8, 1), (4, 1), (8, 4), (16, 4)):
            ctx.set_tiles(angles, 32 if angles else 0, per_warp)
            out = torch.full((g.m,), float("nan"), device="cuda")
            outs.append(P.project(g, xt, out=out))
    finally:
        ctx.set_tiles(0, 0)
    for o in outs[1:]:
        assert torch.equal(o, outs[0])
    assert np.linalg.norm(outs[0].double().cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("geom", GROUPS[1:])
def test_two_image_walk_projects_the_iterate(P, oracle_mod, geom):
    """BA-GMRES with the discrepancy stop projects w_{k+1} and x_k in one walk
    (up to eight angles per warp): its last residual is that of the returned
    iterate (FP32 sums of squares, 1e-6), and a batch, whose walks have their own
    angles per warp, reports the same residuals as one run alone."""
    import torch
    g, og = P.Geometry(*geom), oracle_mod.Geometry(*geom)
    x = np.random.default_rng(13).uniform(0, 1, (g.N, g.N))
    b = oracle_mod.forward(og, x)
    b += 0.3 * np.abs(b).mean() * np.random.default_rng(14).standard_normal(b.shape)
    bt = torch.tensor(b.ravel(), dtype=torch.float32, device="cuda")
    kw = dict(tau=1.0, noise_norm=1e-6)                       # never reached: three steps
    r = P.ba_gmres(g, bt, 3, **kw)
    for res, y in ((r.history[-1], r.x), (r.resnorm, r.x)):
        ref = np.linalg.norm(bt.double().cpu().numpy() - oracle_mod.forward(og, y.double().cpu().numpy().reshape(g.N, g.N)).ravel())
        assert abs(res - ref) <= 1e-5 * ref
    if g.det_spacing >= 1.0:
        probs = [{"geometry": g, "variant": "ba", "maxit": 3, **kw}]
        two = P.Batch(probs + [{"geometry": P.Geometry(16, 4, 23), "variant": "ba", "maxit": 3, **kw}])
        s = two.solve([bt, torch.rand(92, device="cuda")])[0]
        alone = P.Batch(probs).solve([bt])[0]
        assert s.iters == alone.iters and torch.equal(s.x, alone.x)
        assert np.allclose(s.history, r.history, rtol=1e-5)
