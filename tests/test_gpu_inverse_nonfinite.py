"""Off-diagonal entries that are not finite stay out of the rows above them,
in the inverted blocks and in the solve."""
import numpy as np
import pytest

from paper_1612_01855_gb300 import inputs

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(np.asarray(a, dtype=np.float64).T)).cuda().t()


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("row,col", [(20, 3), (13, 2), (9, 8), (31, 0), (30, 17), (16, 15)])
def test_rows_above_stay_finite(cuda_lib, bad, row, col):
    import torch
    import paper_1612_01855_gb300 as g
    n = 32
    L, B = inputs.well_conditioned(n, 4, seed=row)
    good = g.trtri_blocks(_dev(L), n)[0].clone()
    L[row, col] = bad
    Ld = _dev(L)
    inv = g.trtri_blocks(Ld, n)[0]
    assert torch.equal(inv[:row], good[:row])
    assert not torch.isfinite(inv[row, col])
    X = g.trsm_solve(g.trsm_plan(Ld, n), _dev(B))
    assert torch.isfinite(X[:row]).all() and not torch.isfinite(X[row]).any()
