"""The two forms of the FP64 solve (tile tasks, columns in every division of
the work that fits) give the same bits, on ragged last blocks, odd orders and
blocks that are not whole row groups."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1612_01855_gb300 import inputs

pytestmark = pytest.mark.gpu
TOL = 1e-12  # FP64 parity with the oracle, as in the other solve tests


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(np.asarray(a, dtype=np.float64).T)).cuda().t()


def _solve(lib, plan, B, X, S, CW):
    import torch
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    return lib.trsm_solve_form(plan.handle, p(B), B.shape[1], B.stride(1), p(X), X.stride(1), S, CW, s)


@pytest.mark.parametrize("n,n0", [(1, 1), (2, 2), (31, 32), (33, 33), (65, 64), (193, 64), (255, 34), (257, 256),
                                  (510, 100), (777, 64), (1023, 128), (1537, 256)])
@pytest.mark.parametrize("k", [1, 5, 9, 40])
def test_same_bits(cuda_lib, n, n0, k):
    import torch
    import paper_1612_01855_gb300 as g
    L, B = inputs.well_conditioned(n, k, seed=n + k)
    plan = g.trsm_plan(_dev(L), n0)
    Bd = _dev(B)
    want = torch.empty_like(Bd)
    assert _solve(cuda_lib, plan, Bd, want, 0, 0) == 0
    ref = oracle.forward_subst(L, B)
    assert float(np.max(np.abs(want.cpu().numpy() - ref)) / np.max(np.abs(ref))) < TOL
    ran = set()
    for S in range(1, 9):
        for CW in range(1, 9):
            X = torch.full((k, n + 3), float("nan"), dtype=torch.float64, device="cuda").t()[:n]
            rc = _solve(cuda_lib, plan, Bd, X, S, CW)
            if S > plan.nblocks:
                assert rc == -1
            if rc == 0:
                ran.add((S, CW))
                assert torch.equal(X, want), (S, CW)
    # one block row's W and S + 1 of X_b are 2 n0 CW doubles at least
    assert {(S, CW) for S in range(1, min(8, plan.nblocks) + 1) for CW in range(1, 4)} <= ran
    assert torch.equal(g.trsm_solve(plan, Bd), want)
    g.trsm_sync_status(plan)


def test_choice_and_arguments(cuda_lib):
    """The smallest solves run by columns, wide ones as tile tasks; orders the
    column form does not take are refused by it."""
    import paper_1612_01855_gb300 as g

    def choice(plan, k):
        S, CW = ctypes.c_int(-1), ctypes.c_int(-1)
        assert cuda_lib.trsm_solve_form_choice(plan.handle, k, ctypes.byref(S), ctypes.byref(CW)) == 0
        return S.value, CW.value

    L, B = inputs.well_conditioned(600, 3, seed=1)
    small = g.trsm_plan(_dev(L[:64, :64]), 64)
    assert choice(small, 1)[0] == 1
    plan = g.trsm_plan(_dev(L), 64)
    assert choice(plan, 1)[0] > 1 and choice(plan, 200000) == (0, 0)
    Bd = _dev(B)
    for n0 in (33, 257, 300):  # several blocks of odd order; blocks longer than 256
        other = g.trsm_plan(_dev(L), n0)
        assert choice(other, 1) == (0, 0)
        assert _solve(cuda_lib, other, Bd, Bd.clone(), 1, 1) == -1
    for S, CW in ((1, 0), (0, 1), (9, 1), (1, 9), (-1, 2)):
        assert _solve(cuda_lib, plan, Bd, Bd.clone(), S, CW) == -1
    assert cuda_lib.trsm_solve_form(None, None, 1, 1, None, 1, 0, 0, None) == -1
    assert cuda_lib.trsm_solve_form_choice(None, 1, None, None) == -1


@pytest.mark.parametrize("n,n0", [(2, 2), (64, 64), (128, 64), (128, 128), (1000, 64), (1272, 256)])
def test_no_more_columns_a_group_than_there_are(cuda_lib, n, n0):
    """A group wider than the right-hand side would solve columns of zeros."""
    import paper_1612_01855_gb300 as g
    L, _ = inputs.well_conditioned(n, 1, seed=2)
    plan = g.trsm_plan(_dev(L), n0)
    S, CW = ctypes.c_int(-1), ctypes.c_int(-1)
    for k in range(1, 9):
        assert cuda_lib.trsm_solve_form_choice(plan.handle, k, ctypes.byref(S), ctypes.byref(CW)) == 0
        assert S.value >= 1 and 1 <= CW.value <= k, (k, S.value, CW.value)
