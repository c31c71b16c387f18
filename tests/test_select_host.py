"""The certified FP32 selection (teno_cert.cuh, select_diffs) on the host:
where it claims the three delta bits of eq. 2.14, exact rational arithmetic
(eq. 2.8-2.14 with C_T of eq. 3.1-3.4, or a fixed C_T) must give the same
bits.  The claim is exact, so there is no tolerance.  Lines: random shapes
from noise level to shocks, at magnitudes 1e-6 ... 1e6, scaled lines whose
tau/dmin sits at the thresholds of m, and lines of two or three values that
put a stencil's chi at C_T."""
import ctypes
import os
import subprocess
import tempfile
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2003_09145_gb300", "csrc")
H, B_L, B_U, EPS = 10.0, 4, 10, 1e-6


@pytest.fixture(scope="module")
def lib():
    out = os.path.join(tempfile.mkdtemp(prefix="teno_select_host_"), "libselect.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off", f"-I{CSRC}",
                           "-o", out, os.path.join(HERE, "select_host.cpp")])
    return ctypes.CDLL(out)


def thresholds():
    K = B_U - B_L
    return [H * (K / j - 1.0) for j in range(1, K)] + [H * 2.0**-53]


def keep_all_mask():
    bits = 0
    for c, t in enumerate(thresholds()):
        if 3.0 * (1.0 + t) ** 6 * 10.0 ** -(B_L + c + 1) <= 1.0 - 1e-9:
            bits |= 1 << (B_L + c + 1)
    return bits


def exact_select(e, m_fixed):
    e = [Fraction(a) for a in e]
    a = [e[1] - e[0], e[2] - e[1], e[3] - e[2]]
    c = [3 * e[1] - e[0], e[1] + e[2], e[3] - 3 * e[2]]
    D = [Fraction(13, 3) * a[k] ** 2 + c[k] ** 2 + 4 * Fraction(EPS) for k in range(3)]
    tau = abs(D[2] - D[0])
    m = m_fixed
    if m < 0:
        m = B_L + sum(tau <= Fraction(t) * min(D) for t in thresholds())
    g = [((d + tau) / d) ** 6 for d in D]
    ct = Fraction(10.0 ** -m) * sum(g)
    return sum(1 << k for k in range(3) if g[k] >= ct)


def lines(rng, n):
    out = []
    for _ in range(n):
        scale = 10.0 ** rng.uniform(-6, 6)
        kind = rng.integers(4)
        if kind == 0:      # smooth, any steepness
            t = np.arange(5.0) * 10.0 ** rng.uniform(-3, 0.5)
            v = np.sin(t + rng.uniform(0, 6)) + rng.uniform(-1, 1)
        elif kind == 1:    # jump on a smooth line
            v = 10.0 ** rng.uniform(-5, 0) * rng.standard_normal(5) + rng.uniform(-1, 1)
            v[rng.integers(1, 5):] += 10.0 ** rng.uniform(-3, 1)
        elif kind == 2:    # noise on an offset
            v = rng.uniform(-2, 2) + 10.0 ** rng.uniform(-7, 0) * rng.standard_normal(5)
        else:              # a kink: one stencil much smoother than the others
            v = np.array([0, 0, 0, 1.0, rng.uniform(1, 5)]) * 10.0 ** rng.uniform(-4, 0)
            v = v + 10.0 ** rng.uniform(-8, -2) * rng.standard_normal(5)
            if rng.integers(2):
                v = v[::-1]
        out.append(np.ascontiguousarray(v * (scale if rng.integers(2) else 1.0)))
    # lines whose first or last differences put tau/dmin near a threshold of m
    for thr in thresholds()[:-1]:
        for _ in range(n // 20):
            lo, hi = 1e-6, 1e6
            shape = rng.standard_normal(5)
            base = np.array([0.0, 1.0, 2.0, 3.0, 4.0]) * rng.uniform(0.1, 1)
            for _ in range(60):
                mid = np.sqrt(lo * hi)
                v = base + mid * shape
                ee = np.diff(v)
                aa = ee[1:] - ee[:-1]
                cc = np.array([3 * ee[1] - ee[0], ee[1] + ee[2], ee[3] - 3 * ee[2]])
                b = 13 / 3 * aa**2 + cc**2
                lo, hi = (mid, hi) if abs(b[2] - b[0]) < thr * (b.min() + 4 * EPS) else (lo, mid)
            out.append(base + np.sqrt(lo * hi) * (1 + 10.0 ** rng.uniform(-7, -2)) * shape)
    return np.array(out)


@pytest.mark.parametrize("m_fixed", [-1, 5, 7])
def test_certified_selection_is_exact(lib, m_fixed):
    V = np.ascontiguousarray(np.diff(lines(np.random.default_rng(11 + m_fixed), 3000), axis=1))
    out = np.full(len(V), -2, dtype=np.int32)
    thr = np.zeros(16, dtype=np.float32)
    thr[:6] = np.array(thresholds(), dtype=np.float32)
    ct = np.array([10.0**-m for m in range(16)], dtype=np.float32)
    eps4 = np.nextafter(np.float32(4 * EPS), np.float32(0))
    # the keep-all threshold: LAD's j = 3 (m >= 7), or 3 (1 + thr)^6 C_T < 1
    keep = thresholds()[2] if m_fixed < 0 else (0.33 * 10.0**m_fixed) ** (1 / 6) - 1
    keep = np.nextafter(np.float32(keep), np.float32(0))
    ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    lib.select_batch(ctypes.c_int64(len(V)), ptr(V), ctypes.c_float(eps4), ctypes.c_float(keep), ptr(thr), 6, B_L, m_fixed,
                     keep_all_mask() if m_fixed < 0 else 0, ptr(ct), ptr(out))
    decided = np.flatnonzero(out >= 0)
    bad = [i for i in decided if out[i] != exact_select(V[i], m_fixed)]
    assert not bad, (len(bad), V[bad[0]].tolist(), out[bad[0]], exact_select(V[bad[0]], m_fixed))
    # not vacuous: most lines are decided, and every kind of selection occurs
    assert len(decided) > 0.7 * len(V), len(decided) / len(V)
    assert {1, 4, 7} <= set(out[decided].tolist())
