"""The CGS2 step's second pass with one read of the basis (cgs_sweep_kernel),
against the same passes in FP64: ragged lengths, every number of warps to a
stream (k up to 16, 32, 64, 128, 216) at its edges, row strides, w_out in q's
place, two runs' bits, and the first length and k on either side of its range."""
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


SIZES = [(900, 129, 0), (1027, 216, 12), (1027, 217, 4), (2051, 200, 64), (19461, 150, 4), (131072, 130, 0),
         (3125001, 8, 4), (3571430, 7, 0), (1562501, 16, 0), (1470589, 17, 8), (781252, 32, 0), (757577, 33, 4),
         (390627, 64, 0), (3846157, 65, 4), (585938, 128, 0), (4194304, 60, 0)]


@pytest.mark.parametrize("L,k,pad", SIZES)
def test_second_pass_reads_the_basis_once(P, L, k, pad):
    import torch
    torch.manual_seed(L + k)
    ld = (L + 3) // 4 * 4 + pad
    W = torch.full((k, ld), float("nan"), device="cuda")      # nothing beyond L may be read
    W[:, :L] = torch.randn(k, L, device="cuda") / L ** 0.5
    q0 = torch.randn(L, device="cuda")
    q = q0.clone()
    h, w = P.cgs2(W, k, q)
    # FP64, vector by vector: both sweeps and the norm from ||q1|| and h2
    r = q0.double()
    hs = []
    for _ in range(2):
        c = torch.stack([W[j, :L].double() @ r for j in range(k)])
        n2 = float(r @ r)
        for j in range(k):
            r -= c[j] * W[j, :L].double()
        hs.append(c)
        if len(hs) == 1:
            n2 = float(r @ r)
    nrm = (n2 - float(hs[1] @ hs[1])) ** 0.5
    # each of the k terms of an update, each coefficient and each sum is
    # rounded to FP32 once or twice: first order k 2^-24 of ||q||
    tol = (k + 16) * 2.0 ** -24
    nq = float(q0.double().norm())
    assert float((q.double() - r).norm()) <= tol * nq
    assert float((h[:k] - hs[0] - hs[1]).abs().max()) <= tol * nq
    assert abs(float(h[k]) - nrm) <= tol * nq
    assert float((w.double() - r / nrm).norm()) <= 2 * tol * nq / nrm
    # the same bits again, with w_out in q's place
    q2 = q0.clone()
    h2, w2 = P.cgs2(W, k, q2, q2)
    assert torch.equal(h2, h) and torch.equal(w2, w)
