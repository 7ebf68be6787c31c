"""The blocks that small plans pass on: ordinary device memory, bounded while
idle whatever is held beside it, and given on only when no solve is left."""
import ctypes
import threading

import numpy as np
import pytest

import oracle
from paper_1612_01855_gb300 import inputs

pytestmark = pytest.mark.gpu
IPC_CAPABLE = 10  # CU_POINTER_ATTRIBUTE_IS_LEGACY_CUDA_IPC_CAPABLE


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(np.asarray(a, dtype=np.float64).T)).cuda().t()


def _ipc_capable(ptr):
    v = ctypes.c_int(-1)
    rc = ctypes.CDLL("libcuda.so.1").cuPointerGetAttribute(ctypes.byref(v), IPC_CAPABLE, ctypes.c_uint64(ptr))
    assert rc == 0
    return v.value


def _lt(lib, plan):
    ld = ctypes.c_int64()
    p = lib.trsm_plan_lt(plan.handle, ctypes.byref(ld))
    return p if isinstance(p, int) else ctypes.cast(p, ctypes.c_void_p).value


@pytest.mark.parametrize("n", [64, 500])
def test_lt_can_be_shared_like_cudamalloc_memory(cuda_lib, n):
    import torch
    import paper_1612_01855_gb300 as g
    L, _ = inputs.well_conditioned(n, 1, seed=1)
    Ld = _dev(L)
    for _ in range(2):  # a fresh block, then one passed on
        plan = g.trsm_plan(Ld, 64)
        assert _ipc_capable(_lt(cuda_lib, plan)) == _ipc_capable(torch.empty(1 << 22, device="cuda").data_ptr())
        plan.destroy()


def test_destroy_waits_for_the_device(cuda_lib):
    """A block goes on as soon as trsm_destroy returns, so that call has to
    wait for whatever runs, on any stream."""
    import torch
    import paper_1612_01855_gb300 as g
    L, _ = inputs.well_conditioned(500, 1, seed=2)
    plan = g.trsm_plan(_dev(L), 64)
    side = torch.cuda.Stream()
    done = torch.cuda.Event()
    with torch.cuda.stream(side):
        torch.cuda._sleep(100_000_000)  # about 50 ms
        done.record()
    assert not done.query()
    plan.destroy()
    assert done.query()


def test_idle_blocks_stay_beside_many_live_ones_and_are_bounded(cuda_lib):
    import torch
    import paper_1612_01855_gb300 as g
    n = 1800  # 26 MB
    L, _ = inputs.well_conditioned(n, 1, seed=3)
    Ld = _dev(L)
    g.workspace_trim(0)
    torch.cuda.synchronize()
    base = g.workspace_reserved_bytes()
    plans = [g.trsm_plan(Ld, 256) for _ in range(14)]  # 364 MB
    g.workspace_trim(0)
    torch.cuda.synchronize()
    held = g.workspace_reserved_bytes()
    assert held - base >= 14 * 8 * n * n
    plans.pop().destroy()
    torch.cuda.synchronize()
    assert g.workspace_reserved_bytes() == held  # the block stays for the next plan
    plans.append(g.trsm_plan(Ld, 256))
    all_live = g.workspace_reserved_bytes()
    for p in plans:
        p.destroy()
    torch.cuda.synchronize()
    assert g.workspace_reserved_bytes() <= all_live - 14 * 8 * n * n + (256 << 20)
    g.workspace_trim(0)
    torch.cuda.synchronize()
    assert g.workspace_reserved_bytes() <= base


def test_threads(cuda_lib):
    """Plans made, used and destroyed on four threads and streams at once."""
    import torch
    import paper_1612_01855_gb300 as g
    n, k = 200, 3
    sys_ = [inputs.well_conditioned(n, k, seed=10 + i) for i in range(4)]
    want = [oracle.forward_subst(L, B) for L, B in sys_]
    devs = [(_dev(L), _dev(B)) for L, B in sys_]
    torch.cuda.synchronize()
    bad = []

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(25):
                    plan = g.trsm_plan(devs[i][0], 64)
                    X = g.trsm_solve(plan, devs[i][1])
                    plan.destroy()
                    err = float(np.max(np.abs(X.cpu().numpy() - want[i])) / np.max(np.abs(want[i])))
                    if not err < 1e-12:
                        bad.append((i, err))
        except Exception as e:  # noqa: BLE001 - reported below
            bad.append((i, e))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
