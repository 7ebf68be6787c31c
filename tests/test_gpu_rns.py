"""The residue-number-system products under the sliced residual and schedule:
exact integer sums at the largest residues, tile edges, and values that are
not finite."""
import ctypes

import numpy as np
import pytest

from paper_1612_01855_gb300 import inputs

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(np.asarray(a, dtype=np.float64).T)).cuda().t()


def _residual(lib, L, X, B, planes):
    import torch
    n, k = B.shape
    Ld, Xd, Bd = _dev(L), _dev(X), _dev(B)
    Rd = torch.full((k, n), float("nan"), dtype=torch.float64, device="cuda").t()
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert lib.trsm_residual_sliced(p(Ld), n, n, p(Xd), k, n, p(Bd), n, p(Rd), n, planes, p(err), s) == 0
    torch.cuda.synchronize()
    assert err.item() == 0
    return Rd.cpu().numpy()


@pytest.mark.parametrize("planes", [5, 7, 8])
@pytest.mark.parametrize("a,b", [((1 << 47) + 89, (1 << 34) + 89), ((1 << 48) - 1, (1 << 35) - 1),
                                 (0x7FFFC1234567, -0x3F1234567)])
def test_constant_factors_largest_sums(cuda_lib, planes, a, b):
    """Every entry of the strictly lower L equal to one 48-bit integer and
    every entry of X to one 35-bit integer: all residues of a modulus have
    the same sign, so the FP32 sums over a 2048-wide chunk are the largest
    there are.  The exact result is -i a b and the factors are not rounded;
    the integer is put together to M 2^-64 (M < 2^95.6, 2^102.7, 2^109.7 for
    the classes), then each of the two chunks has a few FP64 roundings.  An
    FP32 sum that was not exact would be off by at least M / p > 2^-8 M."""
    n, k = 2200, 3
    L = np.tril(np.full((n, n), float(a)), -1)
    R = _residual(cuda_lib, L, np.full((n, k), float(b)), np.zeros((n, k)), planes)
    # M 2^-64 relative to the class's scale, 2^(48 + bits) = |a| |b| scaled up
    bits, m = {5: (35, 95.6), 7: (42, 102.7), 8: (48, 109.7)}[planes]
    unit = 2.0 ** (m - 64 - (48 + bits)) * 2.0 ** (a.bit_length() + abs(b).bit_length())
    for j in range(k):
        for i in range(1, n):
            want = -i * a * b
            # the cut limbs of the 15 residues add up to 2^-61.5 M at most: 6 units
            assert abs(int(R[i, j]) - want) <= 2 * 7 * unit + (abs(want) >> 50), (i, R[i, j], want)
    assert np.all(R[0] == 0)


@pytest.mark.parametrize("n", [1, 64, 129, 257, 2048, 2049, 4097])
@pytest.mark.parametrize("k", [1, 64, 65, 128, 129, 256, 257])
def test_tile_edges(cuda_lib, n, k):
    """Row tiles of 128 (one CTA) and 256 (a pair), column tiles of 64, 128
    and 256, chunks of 2048.  Both factors carry 48 bits of their (row, chunk)
    maximum: an error of 2^-48 of n times the product of the maxima, here
    within a factor of 8 of |B| + |L| |X|, and numpy's own n 2^-53."""
    L, B = inputs.well_conditioned(n, k, seed=n + k)
    X = np.random.default_rng(n * k).uniform(-1, 1, size=(n, k))
    R = _residual(cuda_lib, L, X, B, 8)
    scale = np.abs(B) + np.abs(np.tril(L)) @ np.abs(X)
    assert np.max(np.abs(R - (B - np.tril(L) @ X)) / scale) < 2.0 ** -45 + n * 2.0 ** -53


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_non_finite_columns_stay_apart(cuda_lib, bad):
    """An infinity or NaN in one column of B leaves the other columns' bits as
    they were, and that column non-finite from its block row on."""
    import torch
    import paper_1612_01855_gb300 as g
    n, k, n0 = 700, 70, 128
    L, B = inputs.well_conditioned(n, k, seed=21)
    plan = g.trsm_plan(_dev(L), n0)
    good = g.trsm_solve_schedule(plan, _dev(B), schedule="sliced").clone()
    B[300, 33] = bad
    X = g.trsm_solve_schedule(plan, _dev(B), schedule="sliced")
    g.trsm_sync_status(plan)
    keep = [j for j in range(k) if j != 33]
    assert torch.equal(X[:, keep], good[:, keep])
    assert torch.equal(X[:256, 33], good[:256, 33])  # the block rows before
    assert not torch.isfinite(X[300:, 33]).any()


def test_two_streams(cuda_lib):
    """Solves on two streams at once give the bits of a solve alone."""
    import torch
    import paper_1612_01855_gb300 as g
    n, k, n0 = 1500, 300, 256
    L, B = inputs.well_conditioned(n, k, seed=4)
    plan = g.trsm_plan(_dev(L), n0)
    Bd = _dev(B)
    want = g.trsm_solve_schedule(plan, Bd, schedule="sliced").clone()
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    outs = [torch.empty_like(Bd) for _ in range(6)]
    for i, X in enumerate(outs):
        with torch.cuda.stream(streams[i % 2]):
            g.trsm_solve_schedule(plan, Bd, X=X, schedule="sliced")
    torch.cuda.synchronize()
    assert all(torch.equal(X, want) for X in outs)
    g.trsm_sync_status(plan)
