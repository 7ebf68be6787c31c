"""The solve by columns (small and narrow FP64 solves): edges of the row
groups, column groups and clusters against the oracle, at the FP64 parity
tolerance of the other schedules."""
import numpy as np
import pytest

import oracle
from paper_1612_01855_gb300 import inputs

pytestmark = pytest.mark.gpu
TOL = 1e-12


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(np.asarray(a, dtype=np.float64).T)).cuda().t()


def _rel(a, b):
    return float(np.max(np.abs(a - b)) / np.max(np.abs(b)))


@pytest.mark.parametrize("n,n0", [(2, 2), (31, 32), (64, 64), (65, 64), (193, 64), (255, 34), (257, 256), (1023, 128),
                                  (1100, 100), (1537, 256)])
@pytest.mark.parametrize("k", [1, 2, 17, 37, 77, 153, 305, 460])
def test_parity(cuda_lib, n, n0, k):
    """Ragged last blocks of odd and even order, blocks that are not whole
    row groups, one to eight columns a group and one to eight CTAs."""
    import paper_1612_01855_gb300 as g
    L, B = inputs.well_conditioned(n, k, seed=n + k)
    p = g.trsm_plan(_dev(L), n0)
    X = g.trsm_solve(p, _dev(B))
    g.trsm_sync_status(p)
    assert _rel(X.cpu().numpy(), oracle.forward_subst(L, B)) < TOL


def test_in_place_layouts_and_streams(cuda_lib):
    """In place, with leading dimensions above n, on two streams at once, and
    with a column that is not finite: the bits of the plain solve in every
    other column."""
    import torch
    import paper_1612_01855_gb300 as g
    n, k, n0 = 777, 45, 64
    L, B = inputs.well_conditioned(n, k, seed=3)
    p = g.trsm_plan(_dev(L), n0)
    Bd = _dev(B)
    want = g.trsm_solve(p, Bd).clone()
    big = torch.full((k, n + 9), float("nan"), dtype=torch.float64, device="cuda")
    Xv = big.t()[:n]
    Xv.copy_(Bd)
    g.trsm_solve(p, Xv, X=Xv)
    assert torch.equal(Xv, want) and torch.isnan(big.t()[n:]).all()
    outs = [torch.empty_like(Bd) for _ in range(6)]
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    for i, X in enumerate(outs):
        with torch.cuda.stream(streams[i % 2]):
            g.trsm_solve(p, Bd, X=X)
    torch.cuda.synchronize()
    assert all(torch.equal(X, want) for X in outs)
    bad = Bd.clone()
    bad[100, 7] = float("nan")
    X = g.trsm_solve(p, bad)
    keep = [j for j in range(k) if j != 7]
    assert torch.equal(X[:, keep], want[:, keep]) and torch.isnan(X[128:, 7]).all()
    g.trsm_sync_status(p)
