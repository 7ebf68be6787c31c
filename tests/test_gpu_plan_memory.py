"""Plans whose memory comes from the library's pool: a block that held another
plan is used again as it was left."""
import numpy as np
import pytest

import oracle
from paper_1612_01855_gb300 import inputs

pytestmark = pytest.mark.gpu


def _dev(A):
    import torch
    return torch.from_numpy(np.ascontiguousarray(A.T)).to("cuda").t()


@pytest.mark.parametrize("n,n0", [(61, 64), (1022, 128), (1999, 256)])
def test_plan_in_reused_memory(cuda_lib, n, n0):
    """Rows n .. ldt - 1 of L~ and everything above the diagonal are not to be
    read as what the last plan left there (not-a-numbers here).  n = 1999 is
    about the largest plan the pool takes (32 MiB)."""
    import torch
    import paper_1612_01855_gb300 as g
    k = 40
    big = (n + 3) // 4 * 4
    bad, _ = inputs.well_conditioned(big, 1, seed=3)
    bad[np.tril_indices(big, -1)] = np.nan
    L, B = inputs.well_conditioned(n, k, seed=4)
    Ld, Bd, badd = _dev(L), _dev(B), _dev(bad)
    want = oracle.forward_subst(L, B)
    scale = float(np.max(np.abs(want)))
    first = g.trsm_plan(badd, n0)
    first.destroy()
    plan = g.trsm_plan(Ld, n0)
    outs = [g.trsm_solve(plan, Bd), g.trsm_solve(plan, Bd[:, :1]),
            g.trsm_solve_schedule(plan, Bd, schedule="sliced")]
    g.trsm_plan_mixed(plan, Ld, inner="fp16x3")
    outs.append(g.trsm_solve_mixed(plan, Bd, tol=1e-13)[0])
    g.trsm_sync_status(plan)
    for X in outs:
        w = want[:, :X.shape[1]]
        # the bound of the library's other solve tests on these inputs
        assert float(np.max(np.abs(X.cpu().numpy() - w))) < 1e-12 * scale
    assert torch.isfinite(outs[0]).all()
    plan.destroy()


def test_destroy_waits_and_memory_is_bounded(cuda_lib):
    """Making and destroying one small plan after another holds no more than
    the first did, trimming gives it back, and a plan destroyed right behind
    its solve leaves the solve's results whole."""
    import torch
    import paper_1612_01855_gb300 as g
    n, k = 1500, 2000
    L, B = inputs.well_conditioned(n, k, seed=5)
    Ld, Bd = _dev(L), _dev(B)
    want = oracle.forward_subst(L, B)
    side = torch.cuda.Stream()
    g.workspace_trim(0)
    torch.cuda.synchronize()
    base = g.workspace_reserved_bytes()
    held = []
    for _ in range(4):
        plan = g.trsm_plan(Ld, 64)
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            X = g.trsm_solve(plan, Bd)
        plan.destroy()
        other = g.trsm_plan(2.0 * Ld, 64)  # takes the same block
        side.synchronize()
        other.destroy()
        held.append(g.workspace_reserved_bytes())
        assert float(np.max(np.abs(X.cpu().numpy() - want))) < 1e-12 * float(np.max(np.abs(want)))
        del X
    assert held[-1] == held[0]
    g.workspace_trim(0)
    torch.cuda.synchronize()
    assert g.workspace_reserved_bytes() <= base
