"""What the performance of this package is measured on.

Each case is the work a user has one call do, through the public entry points
of ``paper_1612_01855_gb300``: FP64 solves with a resident plan from the
smallest request a server sees to the narrow end of the k/n sweep, planning
and the inversion of the diagonal blocks, the sliced schedule, the refined
mixed-precision solve, and batches of uneven systems in both data types.
Sizes are those of the benchmark, its serving and batching workloads and the
tests.  Matrices follow the package's own recipes (diagonal U[2, 3] or graded,
strictly lower part U[-1, 1] / n, B U[-1, 1]), drawn on the device.
"""
import math

import numpy as np
import torch

import paper_1612_01855_gb300 as g

DEV = "cuda"


def listed():
    return [
        # the smallest request of the serving workload: one right-hand side
        # against a resident 64 x 64 plan (pure call and launch latency)
        {"name": "solve_smallest", "kind": "solve", "n": 64, "k": 1, "n0": 64},
        # a mid-size ragged request against a resident plan (a dependency
        # chain of 16 block rows, one and a bit column tiles)
        {"name": "solve_ragged", "kind": "solve", "n": 1000, "k": 37, "n0": 64},
        # the oracle-sized configuration, a new L each time: plan, then solve
        {"name": "plan_solve_512", "kind": "plan_solve", "n": 512, "k": 512, "n0": 64},
        # the narrow end of the k/n sweep in plain FP64
        {"name": "solve_narrow", "kind": "solve", "n": 16384, "k": 256, "n0": 256},
        # the inverted diagonal blocks of a large L on their own
        {"name": "invert_blocks", "kind": "trtri", "n": 8192, "n0": 512},
        # a large request of the serving workload, as its server runs it: the
        # sliced schedule on a plan of 256-row blocks, ragged last block
        {"name": "sliced_serving", "kind": "sliced", "n": 3000, "k": 200, "n0": 256},
        # the two ends of the k/n sweep under the sliced schedule
        {"name": "sliced_narrow", "kind": "sliced", "n": 16384, "k": 256, "n0": 2048},
        {"name": "sliced_square", "kind": "sliced", "n": 8192, "k": 8192, "n0": 2048},
        # a mixed-precision request of the serving workload
        {"name": "mixed_serving", "kind": "mixed", "n": 3000, "k": 128, "n0": 256, "c": 0, "inner": "fp16x3",
         "tol": 1e-12},
        # the precision configuration: graded diagonal, split-fp16 updates,
        # refined to FP64 accuracy
        {"name": "mixed_precision", "kind": "mixed", "n": 16384, "k": 4096, "n0": 1024, "c": 2, "inner": "fp16x3",
         "tol": 1e-11},
        # the batching workload in both data types, one CUDA graph replay each
        {"name": "batch_f64", "kind": "batch", "dtype": "f64", "count": 4096, "nmax": 1024, "kmax": 256},
        {"name": "batch_f32", "kind": "batch", "dtype": "f32", "count": 4096, "nmax": 1024, "kmax": 256},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "plan_solve", "trtri", "sliced", "sliced", "mixed", "batch"])
    if kind in ("solve", "plan_solve"):
        n = _logint(rng, 64, 8192)
        k = _logint(rng, 1, 2048)
        while float(n) * n * k > 6e10:  # the narrow FP64 solve's work
            k = max(1, k // 2)
        return {"kind": kind, "n": n, "k": k, "n0": 256 if n >= 1024 else 64}
    if kind == "trtri":
        return {"kind": kind, "n": _logint(rng, 64, 8192), "n0": rng.choice([64, 128, 256, 512])}
    if kind == "sliced":
        n = _logint(rng, 2048, 16384)
        k = _logint(rng, 8, 8192)
        while float(n) * n * k > 5e11:
            k = k // 2
        return {"kind": kind, "n": n, "k": k, "n0": rng.choice([256, 512, 1024, 2048])}
    if kind == "mixed":
        n = _logint(rng, 2048, 8192)
        k = _logint(rng, 1, 2048)
        inner = rng.choice(["fp16x3", "fp16x3", "tf32"])
        return {"kind": kind, "n": n, "k": k, "n0": rng.choice([256, 512, 1024]), "c": rng.choice([0, 2]),
                "inner": inner, "tol": 1e-11}
    return {"kind": kind, "dtype": rng.choice(["f64", "f32"]), "count": _logint(rng, 64, 2048),
            "nmax": rng.choice([256, 512, 1024]), "kmax": _logint(rng, 16, 256)}


def _gen(seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    return gen


def _rand(gen, rows, cols, dtype=torch.float64):
    """Column-major rows x cols matrix of U[-1, 1]."""
    return torch.rand((cols, rows), generator=gen, device=DEV, dtype=dtype).mul_(2).sub_(1).t()


def _lower(gen, n, c=0, dtype=torch.float64):
    """Column-major lower triangle: strictly lower part U[-1, 1] / n; diagonal
    U[2, 3] (c = 0) or geomspace(1, 10^-c) in a random order."""
    L = _rand(gen, n, n, dtype).t().div_(n).triu_(1)  # row-major view of the transpose
    if c:
        d = torch.logspace(0, -c, n, dtype=dtype, device=DEV)
        d = d[torch.randperm(n, generator=gen, device=DEV)]
    else:
        d = torch.rand(n, generator=gen, device=DEV, dtype=dtype).add_(2)
    L.diagonal().copy_(d)
    return L.t()


def _batch_shapes(case):
    """Sizes of a batch (part of the case, not of its inputs): n log-uniform
    in [32, nmax], k log-uniform in [1, kmax]."""
    rng = np.random.default_rng(1000 + case["count"])
    ns = np.rint(np.exp(rng.uniform(np.log(32), np.log(case["nmax"]), size=case["count"]))).astype(int)
    ks = np.rint(np.exp(rng.uniform(0.0, np.log(case["kmax"]), size=case["count"]))).astype(int)
    return [int(n) for n in ns], [int(k) for k in ks]


def _systems(case, seed):
    dtype = torch.float64 if case["dtype"] == "f64" else torch.float32
    gen = _gen(seed)
    out = []
    for n, k in zip(*_batch_shapes(case)):
        out.append((_lower(gen, n, 0, dtype), _rand(gen, n, k, dtype)))
    return out


def _inputs(case, seed):
    gen = _gen(seed)
    L = _lower(gen, case["n"], case.get("c", 0))
    B = _rand(gen, case["n"], case["k"]) if "k" in case else None
    return L, B


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        # all results in one buffer; 32-row blocks except for large FP64 systems
        pairs = _systems(case, seed)
        X = torch.empty(sum(B.numel() for _, B in pairs), dtype=pairs[0][1].dtype, device=DEV)
        systems, at = [], 0
        for L, B in pairs:
            n, k = B.shape
            systems.append({"L": L, "B": B, "X": X[at:at + n * k].view(k, n).t(),
                            "n0": 32 if case["dtype"] == "f32" or n < 256 else 64})
            at += n * k
        batch = g.Batch(systems, dtype=case["dtype"])
        batch.capture()
        return {"kind": kind, "batch": batch, "X": X, "systems": systems}
    L, B = _inputs(case, seed)
    st = {"kind": kind, "n0": case["n0"], "L": L, "B": B, "plan": None}
    if kind in ("solve", "sliced", "mixed"):
        st["plan"] = g.trsm_plan(L, case["n0"])
        st["X"] = torch.empty_like(B)
    if kind == "plan_solve":
        st["X"] = torch.empty_like(B)
    if kind == "trtri":
        st["inv"] = torch.empty((-(-case["n"] // case["n0"]), case["n0"], case["n0"]), dtype=torch.float64, device=DEV)
    if kind == "sliced":
        g.trsm_plan_sliced(st["plan"])
    if kind == "mixed":
        g.trsm_plan_mixed(st["plan"], L, case["inner"])
        st["tol"] = case["tol"]
    return st


def run(st):
    kind = st["kind"]
    if kind == "batch":
        st["batch"].launch_graph()
        return st["X"]
    if kind == "solve":
        return g.trsm_solve(st["plan"], st["B"], X=st["X"])
    if kind == "sliced":
        return g.trsm_solve_schedule(st["plan"], st["B"], X=st["X"], schedule="sliced")
    if kind == "mixed":
        # the server's settings: adaptive residual, two tf32 planes per factor
        # in the diagonal multiplies
        return g.trsm_solve_mixed(st["plan"], st["B"], X=st["X"], residual="adaptive", tol=st["tol"], s_tc=True,
                                  s_tc_planes=2)[0]
    if kind == "trtri":
        return g.trtri_blocks(st["L"], st["n0"], out=st["inv"])
    # a new plan: the previous one is released first, as when a program
    # replaces its factor
    if st["plan"] is not None:
        st["plan"].destroy()
    st["plan"] = g.trsm_plan(st["L"], st["n0"])
    return g.trsm_solve(st["plan"], st["B"], X=st["X"])


def work(case):
    """Each input read once and each output written once (lower triangles);
    flops of L X = B are n^2 k, of inverting a block of order m m^3 / 3."""
    kind = case["kind"]
    if kind == "batch":
        ns, ks = _batch_shapes(case)
        e = 8 if case["dtype"] == "f64" else 4
        return {"bytes": float(sum(e * (n * n / 2 + 2 * n * k) for n, k in zip(ns, ks))),
                "flops": float(sum(n * n * k for n, k in zip(ns, ks)))}
    n, n0 = case["n"], min(case["n0"], case["n"])
    inv = n * n0 * n0 / 3.0
    if kind == "trtri":
        return {"bytes": 8.0 * n * n0 * 1.5, "flops": inv}
    solve = {"bytes": 8.0 * (n * n / 2 + 2 * n * case["k"]), "flops": float(n) * n * case["k"]}
    if kind == "plan_solve":
        solve["flops"] += inv
    return solve


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return torch.cat([torch.linalg.solve_triangular(L.double(), B.double(), upper=False).t().reshape(-1)
                          for L, B in _systems(case, seed)])
    L, B = _inputs(case, seed)
    if kind != "trtri":
        return torch.linalg.solve_triangular(L, B, upper=False)
    # block b's inverse in the leading corner of out[b], zeros elsewhere
    n, n0 = case["n"], case["n0"]
    out = torch.zeros((-(-n // n0), n0, n0), dtype=L.dtype, device=DEV)
    for b, s in enumerate(range(0, n, n0)):
        m = min(n0, n - s)
        out[b, :m, :m] = torch.linalg.solve_triangular(L[s:s + m, s:s + m], torch.eye(m, dtype=L.dtype, device=DEV),
                                                       upper=False)
    return out
