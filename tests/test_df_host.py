"""teno_df.cuh (numbers as the sum of two binary32 values) on the host,
against exact rationals.  The bounds follow the header's operation counts:
the conversion truncates at 2^-46 of the value; an addition rounds its low
part twice (2 2^-24 of low parts below 2^-22 of the larger operand); a product
loses l_a l_b and three roundings of low parts; the reciprocals lose e^3 of
their seeds (2^-60) and the low part's roundings.  2^-44 of the operands'
scale covers each (2^-43 for the reciprocals, whose low part takes the
conversion's error too)."""
import ctypes
import os
import subprocess
import tempfile
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2003_09145_gb300", "csrc")


@pytest.fixture(scope="module")
def lib():
    out = os.path.join(tempfile.mkdtemp(prefix="teno_df_host_"), "libdf.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off", f"-I{CSRC}",
                           "-o", out, os.path.join(HERE, "df_host.cpp")])
    return ctypes.CDLL(out)


def _values(rng, n, lo, hi):
    v = rng.uniform(1.0, 2.0, n) * 2.0 ** rng.integers(lo, hi, n) * rng.choice([-1.0, 1.0], n)
    # mantissas at the split's edges, and neighbours of powers of two
    m = v.view(np.uint64).copy()
    m[::7] &= ~np.uint64((1 << 29) - 1)
    m[1::7] |= np.uint64((1 << 29) - 1)
    m[2::7] &= ~np.uint64((1 << 52) - 1)
    m[3::7] |= np.uint64((1 << 52) - 1)
    return m.view(np.float64)


def _run(lib, op, a, b):
    out = np.zeros((len(a), 3))
    p = lambda x: x.ctypes.data_as(ctypes.c_void_p)
    lib.df_batch(ctypes.c_int(op), ctypes.c_int64(len(a)), p(a), p(b), p(out))
    return out


F = Fraction


@pytest.mark.parametrize("op", [0, 1, 2, 3, 4, 6])
def test_operations(lib, op):
    rng = np.random.default_rng(op)
    a, b = _values(rng, 4000, -30, 31), _values(rng, 4000, -30, 31)
    if op in (3, 4):
        a = np.abs(a)
    b[::5] = -a[::5] * (1 + rng.standard_normal(len(a[::5])) * 1e-6)      # cancelling sums
    out = _run(lib, op, a, b)
    for x, y, (h, l, d) in zip(a, b, out):
        fx, fy, got = F(float(x)), F(float(y)), F(float(h)) + F(float(l))
        if op == 0:
            want, scale, tol = fx, abs(fx), F(1, 2**46)
        elif op == 1:
            want, scale, tol = fx + fy, max(abs(fx), abs(fy)), F(1, 2**44)
        elif op in (2, 6):
            want = fx * (fy if op == 2 else fx)
            scale, tol = abs(want), F(1, 2**44)
        elif op == 3:
            want = 1 / fx
            scale, tol = want, F(1, 2**43)
        else:
            # (h + l)^2 x = 1 within twice the relative tolerance
            want, got, scale, tol = F(1), got * got * fx, F(1), F(1, 2**42)
        assert abs(got - want) <= scale * tol, (op, x, y, h, l)
        # to_double: the moved low part (up to an ulp of h, 2^-23) rounds once in
        # binary32, 2^-47; its bits below 2^-52 are dropped
        s = F(float(h)) + F(float(l))
        assert abs(F(float(d)) - s) <= abs(s) * F(1, 2**46) + F(1, 2**99), (op, x, y, h, l, d)


def test_small_and_zero(lib):
    a = np.array([0.0, -0.0, 1e-40, -1e-300, 2.0**-101])
    out = _run(lib, 0, a, a)
    assert np.all(np.abs(out[:, 0]) <= 2.0**-100 * (1 + 2.0**-20)) and np.all(np.abs(out[:, 1]) <= 2.0**-122)


def test_fixed_sums(lib):
    """A 2^(E - 1078): exact to 2^-46 of the value for any int64 sum."""
    rng = np.random.default_rng(5)
    n = 4000
    A = (rng.integers(-2**62, 2**62, n) >> rng.integers(0, 62, n)).astype(np.int64)
    A[:8] = [0, 1, -1, 2**62, -2**62, (1 << 42) - 1, -(1 << 42), (1 << 21) - 1]
    E = rng.integers(993, 1118, n).astype(np.uint32)
    out = np.zeros((n, 2))
    p = lambda x: x.ctypes.data_as(ctypes.c_void_p)
    lib.df_fixed(ctypes.c_int64(n), p(A), p(E), p(out))
    for a, e, (h, l) in zip(A.tolist(), E.tolist(), out):
        want = F(a) * (F(2) ** (e - 1078))
        assert abs(F(float(h)) + F(float(l)) - want) <= abs(want) * F(1, 2**46), (a, e, h, l)


def test_zero_is_zero(lib):
    a = np.array([0.0, -0.0, 2.0**-1000, -(2.0**-101), 2.0**-100])
    out = _run(lib, 0, a, a)
    assert np.all(out[:4] == 0.0) and out[4, 0] == 2.0**-100 and out[4, 1] == 0.0


def test_to_double_of_small_values(lib):
    """Down to the end of binary32's normal range: h rounds nothing, l is cut
    at 2^-46 of h, and bits of l below 2^-126 are lost."""
    rng = np.random.default_rng(9)
    a = _values(rng, 6000, -124, -30)
    b = a * (2.0**-25 * rng.uniform(-1, 1, len(a)))
    for op in (5, 1):
        for x, y, (h, l, d) in zip(a, b, _run(lib, op, a, b)):
            s = F(float(h)) + F(float(l))
            assert abs(F(float(d)) - s) <= abs(s) * F(1, 2**46) + F(1, 2**125), (op, x, y, h, l, d)
