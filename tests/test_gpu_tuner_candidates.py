"""The tile autotuner times each kernel once: pass sizes of the back projector
that launch the same kernel share one time."""
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


@pytest.mark.parametrize("geom,forms", [
    ((201, 130, 285, 0, 180, 1.0), 1),       # 2 x 2 blocks
    ((201, 130, 407, 0, 180, 0.7), 2),       # one pixel at a time: 16 or 32 angles per pass, 64 as 32
    ((201, 130, 1138, 0, 180, 0.25), 1),     # its windows leave room for 8
    ((61, 130, 1726, 0, 180, 0.05), 1),      # too wide for shared memory
])
def test_equal_candidates_share_their_time(P, geom, forms):
    import torch
    t = P.Context.get(torch.device("cuda", 0)).tuning(P.Geometry(*geom))
    us = t["back_us"]
    assert all(v > 0 for v in us.values())
    assert us[64] == us[32]
    if forms == 1:
        assert us[16] == us[32] and t["back_chunk"] == 32
    else:
        assert t["back_chunk"] in (16, 32)
