"""The integer products of the sliced residual: short factors (nine 6-bit
digits in a pair) give the one double next to the product, others are off by
at most 3.2 M 2^-64 on the integer scale, to either side alike."""
import ctypes
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
BITS = {5: 35, 7: 42, 8: 48}  # of X's factors; L's have 48
LOG2M = {5: 95.6, 7: 102.7, 8: 109.7}  # of the product M of the class's moduli


def _zero_digits(v, bits):
    """6-bit digits that end v, as an integer of `bits` bits, in zeros."""
    v = abs(v)
    return min(7, (bits - v.bit_length() + (v & -v).bit_length() - 1) // 6) if v else 0


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
@pytest.mark.parametrize("n", [2, 130, 2100])
def test_integer_systems(cuda_lib, planes, n):
    """Integers of 16 bits: every factor is held exactly and every sum is an
    integer below 2^42, so B - L X comes out as that integer, over two chunks
    as well."""
    rng = np.random.default_rng(n + planes)
    L = np.tril(rng.integers(-2 ** 15, 2 ** 15, size=(n, n)))
    X = rng.integers(-2 ** 15, 2 ** 15, size=(n, 5))
    B = rng.integers(-2 ** 40, 2 ** 40, size=(n, 5))
    L[1, 0], X[0, 0] = 3, 5
    R = _residual(cuda_lib, L, X, B, planes)
    assert np.array_equal(R, (B - L @ X).astype(np.float64))


@pytest.mark.parametrize("planes", [5, 7, 8])
def test_single_products(cuda_lib, planes):
    """R(i, j) = -a_i b_j for a_i of up to 48 bits and b_j of up to the class's
    bits, of all lengths and both signs.  Long pairs: the bound, the final
    roundings (2^-52), and a mean error that is not one-sided: the roundings at
    2^-64 and of the result, both uniform, have a standard deviation below 0.5
    units, so that 1/8 of a unit is more than 20 standard errors of 10000 pairs
    (limbs that are cut make it -0.49)."""
    rng = np.random.default_rng(planes)
    n, k = 130, 300
    a = [int(v) >> int(s) for v, s in zip(rng.integers(-2 ** 48, 2 ** 48, size=n), rng.integers(0, 48, size=n))]
    b = [int(v) >> int(s) for v, s in zip(rng.integers(-2 ** BITS[planes], 2 ** BITS[planes], size=k),
                                         rng.integers(0, BITS[planes], size=k))]
    L, X = np.zeros((n, n)), np.zeros((n, k))
    L[1:, 0], X[0] = a[1:], b
    R = _residual(cuda_lib, L, X, np.zeros((n, k)), planes)
    short, off = 0, []
    for i in range(1, n):
        for j in range(k):
            want, got = -(a[i] * b[j]), R[i, j]
            if a[i] == 0 or b[j] == 0:
                assert got == 0
            elif _zero_digits(a[i], 48) + _zero_digits(b[j], BITS[planes]) >= 7:
                short += 1
                assert got == float(want), (a[i], b[j])
            else:
                scale = 2.0 ** (abs(a[i]).bit_length() + abs(b[j]).bit_length() - 48 - BITS[planes])
                unit = 2.0 ** (LOG2M[planes] - 64) * scale
                d = float(Fraction(got) - want)
                assert abs(d) <= 3.2 * unit + abs(want) * 2.0 ** -52, (a[i], b[j])
                off.append(d / unit)
    assert short > 10000 and len(off) > 10000
    assert abs(np.mean(off)) < 0.125


@pytest.mark.parametrize("planes", [5, 7, 8])
def test_cancellation_and_range(cuda_lib, planes):
    """Sums that cancel leave B as it is; products beyond the normal range
    become the subnormal, zero or infinity that FP64 has for them."""
    a, b = [], []
    for p, q in [(-600, -470), (-600, -600), (900, 100), (600, 500), (-500, 480), (-1020, 1000)]:
        a.append(3.0 * 2.0 ** p)
        b.append(5.0 * 2.0 ** q)
    m = len(a)
    n = 2 * m + 1
    L, X = np.zeros((n, n)), np.zeros((n, m))
    X[0] = X[1] = b
    for i in range(m):
        L[2 + i, 0] = a[i]
    L[n - 1, 0], L[n - 1, 1] = 7.0, -7.0
    B = np.zeros((n, m))
    B[n - 1] = np.arange(1.0, m + 1)
    with np.errstate(over="ignore", under="ignore"):
        want = B - np.multiply.outer(L[:, 0], X[0]) - np.multiply.outer(L[:, 1], X[1])
    want[n - 1] = B[n - 1]
    R = _residual(cuda_lib, L, X, B, planes)
    assert np.array_equal(R, want)


def test_six_plane_class_keeps_36_bits(cuda_lib):
    """Six digits are 36 bits: columns of 36-bit integers under an L of +-1
    (seven digits a pair) come out exactly."""
    rng = np.random.default_rng(6)
    n, k = 70, 9
    L = np.tril(rng.choice([-1, 1], size=(n, n)))
    X = rng.integers(-2 ** 36 + 1, 2 ** 36, size=(n, k)) | 1
    B = rng.integers(-2 ** 40, 2 ** 40, size=(n, k))
    R = _residual(cuda_lib, L, X, B, 6)
    assert np.array_equal(R, (B - L @ X).astype(np.float64))
