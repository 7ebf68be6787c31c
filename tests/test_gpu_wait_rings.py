"""The waits of the copy rings and of clusters run out as the others do: the
kernel gives up, drains its copies and returns, and the device stays usable."""
import ctypes
import time

import numpy as np
import pytest

import oracle
from paper_1612_01855_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", [3, 4])  # copy ring, cluster
@pytest.mark.parametrize("limit_us", [1, 50_000])
def test_wait_runs_out_and_device_stays_usable(cuda_lib, kind, limit_us):
    import torch
    import paper_1612_01855_gb300 as g
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    t0 = time.perf_counter()
    assert cuda_lib.trsm_wait_selftest(kind, limit_us, s) == -5  # TRSM_ETIMEOUT
    dt = time.perf_counter() - t0
    assert 0.9e-6 * limit_us <= dt < 2.0
    L, B = inputs.well_conditioned(300, 7, seed=kind)
    Ld = torch.from_numpy(np.ascontiguousarray(L.T)).cuda().t()
    Bd = torch.from_numpy(np.ascontiguousarray(B.T)).cuda().t()
    p = g.trsm_plan(Ld, 64)
    X = g.trsm_solve(p, Bd)
    g.trsm_sync_status(p)
    want = oracle.forward_subst(L, B)
    assert np.max(np.abs(X.cpu().numpy() - want)) <= 1e-12 * np.max(np.abs(want))
