"""The back projector's tiles that share work between a pixel and its point
reflection, and its 2 x 2 pixel blocks: edges of tiles and blocks, the middle
row of an odd image, pitches on both sides of one pixel (blocks or one pixel at
a time), every quadrant of angles, and values that are not finite."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# Per interpolation the position is off by at most 4 ulp(32) / 2 ~ 8e-6 bins and
# the sums by a few 2^-24, each on terms of the data's size, so the relative
# 2-norm error is below 8e-6; 1e-5 is also the projectors' parity bound.
TOL = 1e-5

GEOMS = [
    # N, n_angles, n_det, start, range, det_spacing
    (1, 7, 3, 0, 180, 1.0),           # one pixel: its own reflection
    (2, 5, 4, 0, 360, 1.0),
    (31, 33, 45, 0, 180, 1.0),        # one ragged tile; a CTA's last angles alone in their chunk
    (32, 128, 46, 0, 180, 1.0),       # full chunks exactly
    (33, 129, 50, -45, 90, 1.0),      # middle row shared by a pixel and its reflection; cos >= 0 throughout
    (65, 40, 92, 90, 180, 1.0),       # cos <= 0, then sin < 0
    (63, 24, 30, 7, 360, 2.0),        # all quadrants, the corner changes side inside a chunk; short detector
    (64, 50, 91, 0, 180, 1.001),      # just coarser than a pixel
    (64, 50, 92, 0, 180, 0.999),      # just finer: one pixel at a time
    (47, 30, 300, 0, 180, 0.25),      # fine pitch: windows that allow 8 angles per pass
    (700, 20, 990, 0, 180, 1.0),      # 64-row tiles
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
def test_back_parity_at_tile_edges(P, oracle_mod, geom):
    import torch
    g, og = P.Geometry(*geom), oracle_mod.Geometry(*geom)
    b = np.random.default_rng(5).standard_normal(g.m).astype(np.float32)
    out = torch.full((g.n,), float("nan"), device="cuda")          # every pixel has to be written
    got = P.backproject(g, torch.tensor(b, device="cuda"), out=out).double().cpu().numpy()
    ref = oracle_mod.backproject(og, b.astype(np.float64))
    assert np.linalg.norm(got - ref) <= TOL * np.linalg.norm(ref)
    assert np.abs(got - ref).max() <= 10 * TOL * np.abs(ref).max()


@pytest.mark.parametrize("model,tau", [("matched", 0.0), ("threshold", 0.1)])
@pytest.mark.parametrize("N", [32, 33, 70])
def test_matched_tiles_reach_every_pixel(P, oracle_mod, N, model, tau):
    """A^T against the adjoint of the forward projector, row by row of the
    identity on the detector; B_tau equals A^T where no weight is near the
    threshold (checked through a sinogram of ones against its own sum)."""
    import torch
    g = P.Geometry(N, 21, N + 9, 0, 360, 1.0, back_model=model, back_tau=tau)
    A = oracle_mod.matrix_A(oracle_mod.Geometry(N, 21, N + 9, 0, 360, 1.0))
    b = np.random.default_rng(6).uniform(0.5, 1.0, g.m).astype(np.float32)
    out = torch.full((g.n,), float("nan"), device="cuda")
    got = P.backproject(g, torch.tensor(b, device="cuda"), out=out).double().cpu().numpy()
    ref = np.asarray(A.T @ b.astype(np.float64)).ravel()
    assert np.isfinite(got).all()
    if model == "matched":
        assert np.linalg.norm(got - ref) <= TOL * np.linalg.norm(ref)
    else:
        # only weights below tau max(A) = 0.1 * sqrt(2) are dropped: at most two terms per angle
        assert (got <= ref + 1e-4).all() and (got >= ref - 21 * 2 * 0.1 * np.sqrt(2.0)).all()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_bad_bin_reaches_only_the_pixels_that_interpolate_it(P, oracle_mod, bad):
    import torch
    geom = (65, 40, 92, 0, 180, 1.0)
    g, og = P.Geometry(*geom), oracle_mod.Geometry(*geom)
    b = np.random.default_rng(7).standard_normal(g.m).astype(np.float32)
    ref = oracle_mod.backproject(og, b.astype(np.float64))
    b[13 * 92 + 40] = bad
    got = P.backproject(g, torch.tensor(b, device="cuda")).double().cpu().numpy()
    th = 13 * np.pi / 40
    c = np.arange(65) - 32.0
    u = c[None, :] * np.cos(th) + c[:, None] * np.sin(th) + 45.5
    touched = (np.abs(u - 40) < 1.0).ravel()
    clear = np.abs(np.abs(u - 40) - 1.0).ravel() > 1e-4            # away from the edge of the bin's reach
    assert np.array_equal(~np.isfinite(got)[clear], touched[clear])
    keep = np.isfinite(got)
    assert np.linalg.norm((got - ref)[keep]) <= TOL * np.linalg.norm(ref[keep])


def test_sixteen_bit_basis_column(P, oracle_mod):
    """AB-GMRES back-projects columns of a 16-bit basis: its first Hessenberg
    column reproduces A B w_1 for the stored w_1."""
    import torch
    geom = (50, 33, 71, 0, 180, 1.0)
    g, og = P.Geometry(*geom), oracle_mod.Geometry(*geom)
    b = torch.tensor(np.random.default_rng(8).uniform(0, 1, g.m), dtype=torch.float32, device="cuda")
    for basis, u in (("fp16", 2.0 ** -11), ("bf16", 2.0 ** -8)):
        r = P.ab_gmres(g, b, 1, basis=basis, keep_workspace=True)
        W = r.basis(g, "ab", 1).double().cpu().numpy()
        h = r.hessenberg(g, "ab", 1).cpu().numpy()[:, 0]
        q = oracle_mod.forward(og, oracle_mod.backproject(og, W[0]).reshape(50, 50))
        assert np.linalg.norm(q - W.T @ h) <= 2 * u * np.linalg.norm(q)


@pytest.mark.parametrize("geom", [(47, 70, 100, 0, 180, 0.7), (1030, 40, 2100, 0, 180, 0.75)])
def test_staged_chunk_does_not_change_the_result(P, oracle_mod, geom):
    """Pitches below a pixel, 16 or 32 angles staged per pass, with eight and
    with two CTAs per tile."""
    import torch
    g, og = P.Geometry(*geom), oracle_mod.Geometry(*geom)
    b = np.random.default_rng(10).standard_normal(g.m).astype(np.float32)
    bt = torch.tensor(b, device="cuda")
    ctx = P.Context.get(bt.device)
    try:
        outs = []
        for chunk in (16, 32, 64):
            ctx.set_tiles(8, chunk)
            outs.append(P.backproject(g, bt))
    finally:
        ctx.set_tiles(0, 0)
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[1], outs[2])
    ref = oracle_mod.backproject(og, b.astype(np.float64))
    assert np.linalg.norm(outs[0].double().cpu().numpy() - ref) <= TOL * np.linalg.norm(ref)


@pytest.mark.parametrize("N,Na", [(1024, 60), (1024, 130), (700, 50), (512, 250)])
def test_few_angles_take_smaller_clusters(P, oracle_mod, N, Na):
    import torch
    Nd = int(np.ceil(np.sqrt(2) * N))
    g, og = P.Geometry(N, Na, Nd), oracle_mod.Geometry(N, Na, Nd)
    b = np.random.default_rng(11).standard_normal(g.m).astype(np.float32)
    got = P.backproject(g, torch.tensor(b, device="cuda")).double().cpu().numpy()
    ref = oracle_mod.backproject(og, b.astype(np.float64))
    assert np.linalg.norm(got - ref) <= TOL * np.linalg.norm(ref)
