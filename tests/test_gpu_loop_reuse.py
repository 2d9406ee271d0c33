"""One captured solver loop serves every set of vectors and stopping targets of
its setting: solves in turn with new buffers, targets and start images must give
the bits of the host-driven steps, also where the loop has only some of its
parts (few iterations: no loop of separate passes)."""
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


# the back projector's kernels: blocks, pixel pairs, matched pairs and its general form
BACK = {"blocks": dict(), "pairs": dict(det_spacing=0.8), "threshold": dict(back_model="threshold", back_tau=0.3),
        "matched": dict(back_model="matched", det_spacing=0.25)}


@pytest.mark.parametrize("back", sorted(BACK))
@pytest.mark.parametrize("variant", ["ab", "ba"])
@pytest.mark.parametrize("N,Na,maxit", [(40, 30, 1), (40, 30, 24), (40, 30, 25), (96, 90, 70)])
def test_solves_in_turn_equal_host_driven_steps(P, oracle_mod, variant, N, Na, maxit, back):
    import torch
    from paper_2110_01481_gb300 import inputs as I
    pitch = BACK[back].get("det_spacing", 1.0)
    g = P.Geometry(N, Na, I.detector_count(N), **BACK[back])
    og = oracle_mod.Geometry(N, Na, I.detector_count(N), 0.0, 180.0, pitch)
    fn = P.ab_gmres if variant == "ab" else P.ba_gmres
    clean = oracle_mod.forward(og, I.random_ellipses(N, 7300))
    ctx = P.Context.get(torch.device("cuda", 0))
    ws = torch.empty(P.workspace_bytes(g, variant, maxit), dtype=torch.uint8, device="cuda")
    keep = []                                     # new addresses each time
    for i in range(4):
        b, enorm = I.add_noise(clean, 0.02 * (i + 1), 7301 + i)
        bt = torch.tensor(b.astype(np.float32), device="cuda")
        x0 = None if i % 2 == 0 else torch.full((g.n,), 0.1 * i, device="cuda")
        opts = dict(x0=x0, tau=1.0 + 0.1 * i, noise_norm=None if i == 2 else enorm)
        got = [fn(g, bt, maxit, **opts), fn(g, bt, maxit, workspace=ws, **opts)]
        try:
            ctx.set_timing(True)
            ref = fn(g, bt, maxit, **opts)
        finally:
            ctx.set_timing(False)
            ctx.timing(reset=True)
        for r in got:
            assert (r.iters, r.stop_reason, r.resnorm, r.rho) == (ref.iters, ref.stop_reason, ref.resnorm, ref.rho)
            assert torch.equal(r.x, ref.x) and r.history == ref.history
        res = oracle_mod.forward(og, ref.x.double().cpu().numpy().reshape(N, N)).ravel() - b.ravel()
        assert abs(np.linalg.norm(res) - ref.resnorm) <= 1e-4 * np.linalg.norm(b)
        keep += [bt, x0, got, ref]
