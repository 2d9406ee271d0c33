"""The two forms of a batched CGS2 step, one launch or separate passes, give the
same bits: a batch (one-launch steps) and an engine (separate passes) return
equal iterates, for lengths below, at and above a block's slice and for every
basis type."""
import numpy as np
import pytest

from paper_2110_01481_gb300 import inputs as I

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


@pytest.mark.parametrize("N,Na,basis", [(16, 9, "fp32"), (64, 45, "fp32"), (65, 44, "fp32"), (128, 60, "fp32"),
                                        (64, 45, "fp16"), (65, 44, "bf16")])
def test_passes_equal_the_one_launch_step(P, N, Na, basis):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(N)
    probs, bs = [], []
    for v in ("ab", "ba"):
        g = P.Geometry(N, Na, I.detector_count(N))
        x = torch.rand(g.n, device="cuda", generator=gen)
        b = P.project(g, x)
        b = b + 0.01 * b.abs().mean() * torch.randn(g.m, device="cuda", generator=gen)
        probs.append({"geometry": g, "variant": v, "maxit": 12, "basis": basis})
        bs.append(b)
    batch = P.Batch(probs).solve(bs)
    eng = P.Engine(4, 1 << 33)
    for i, (p, b) in enumerate(zip(probs, bs)):
        assert eng.submit(p["geometry"], b, p["variant"], 12, tag=i, basis=basis) == i
    served = dict(eng.drain(rounds=5))
    for i, r in enumerate(batch):
        assert served[i].iters == r.iters and served[i].history == r.history
        assert torch.equal(served[i].x, r.x), (probs[i]["variant"], basis)
