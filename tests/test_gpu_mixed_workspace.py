"""The refined solve with the FP64 residual holds no residues."""
import numpy as np
import pytest

from paper_1612_01855_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_fp64_residual_workspace(cuda_lib):
    """R, D and W take 20 n k bytes, the operands of one block row at most 16
    n0 k; the residues of X, 30 n k, would not fit in the 64 MiB allowed for
    the rest (the pool maps memory in steps)."""
    import torch
    import paper_1612_01855_gb300 as g
    n, k, n0 = 2048, 4096, 256
    L, B = inputs.well_conditioned(n, k, seed=4)
    Ld = torch.from_numpy(np.ascontiguousarray(L.T)).cuda().t()
    Bd = torch.from_numpy(np.ascontiguousarray(B.T)).cuda().t()
    plan = g.trsm_plan(Ld, n0)
    g.trsm_plan_mixed(plan, Ld, "fp16x3")
    torch.cuda.synchronize()
    g.workspace_trim(0)
    base = g.workspace_reserved_bytes()
    X, _, _ = g.trsm_solve_mixed(plan, Bd, residual="fp64", tol=1e-12, s_tc=True)
    held = g.workspace_reserved_bytes() - base
    assert held <= 20 * n * k + 16 * n0 * k + (64 << 20)
    assert torch.equal(X, g.trsm_solve_mixed(plan, Bd, residual="fp64", tol=1e-12, s_tc=True)[0])
    plan.destroy()
