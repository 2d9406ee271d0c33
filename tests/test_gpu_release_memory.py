"""The workspace memory that a context keeps between solves is given back on
request, and solves before and after give the same bits."""
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


def test_kept_workspace_is_given_back(P):
    import torch
    g = P.Geometry(256, 360, 363)
    maxit = 250
    ws = P.workspace_bytes(g, "ab", maxit)
    assert 100 << 20 < ws < 500 << 20                 # kept, and more than an allocation's granularity
    b = torch.rand(g.m, device="cuda")
    ctx = P.Context.get(b.device)
    ctx.release_memory()                              # whatever earlier solves left
    first = P.ab_gmres(g, b, maxit, tau=1.0, noise_norm=0.5 * float(b.norm()))
    torch.cuda.synchronize()
    kept = torch.cuda.mem_get_info()[0]
    ctx.release_memory()
    ctx.release_memory()                              # nothing left: no harm
    assert torch.cuda.mem_get_info()[0] - kept >= ws - (64 << 20)
    again = P.ab_gmres(g, b, maxit, tau=1.0, noise_norm=0.5 * float(b.norm()))
    assert torch.equal(first.x, again.x) and first.history == again.history
