"""The certificate as the flux passes run it, on the host against exact arithmetic:
the binary32 planes' rounding (near_float), the Roe state in two binary32 values
(roe_df, cert_begin_df), the bound of rounded inputs (kCertRounded) and the paired
test (certify_open2).

Every reconstruction that the mask leaves out must satisfy tau_5 <= thr (min beta_k +
eps) with the binary64 evaluations' margin, for the split values formed exactly from
the binary64 states and the exact Roe average (whose binary64 evaluation the margin
covers).  The interfaces are test_cert_host's, scaled so that one field sits at the
threshold, up to Mach numbers beyond the two-binary32 form's, with the seeds moved by
as much as the hardware's may be off."""
import ctypes
import os
import subprocess
import tempfile
from fractions import Fraction as F

import numpy as np
import pytest

import test_cert_host as tc
import test_closed_host as th

HERE = os.path.dirname(os.path.abspath(__file__))
EPS = 1e-6


def _compile(name):
    out = os.path.join(tempfile.mkdtemp(prefix="teno_cert_rounded_"), "lib.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off", f"-I{th.CSRC}",
                           "-o", out, os.path.join(HERE, name)])
    return ctypes.CDLL(out)


@pytest.fixture(scope="module")
def lib():
    return _compile("closed_host.cpp")


def _exact_roe(sr, sh, su, ndim):
    S = F(float(sr[0])) + F(float(sr[1]))
    u = [(F(float(su[0, k])) + F(float(su[1, k]))) / S for k in range(ndim)]
    q2 = sum(x * x for x in u)
    c2 = F(th.GM1) * ((F(float(sh[0])) + F(float(sh[1]))) / S - q2 / 2)
    hb1 = F(th.GM1) / 2 / c2
    return u, hb1, hb1 * q2 / 2, 1 / (2 * th.root(c2))


def _cases(ndim, d, thr):
    rng = np.random.default_rng(500 + 10 * ndim + d)
    out = []
    for i in range(60):
        vmax = (20.0, 0.8, 6.0)[i % 3]
        base = (rng.uniform(0.5, 2.0), rng.uniform(-vmax, vmax, ndim), rng.uniform(0.5, 2.0))
        pert = rng.standard_normal((6, ndim + 2))
        if i % 2:
            t = np.arange(6.0)[:, None]
            pert = rng.standard_normal((1, ndim + 2)) * t + 0.2 * rng.standard_normal((1, ndim + 2)) * t * t
        pert = pert / np.abs(pert).max()
        scale = (10.0 ** rng.uniform(-4, 4), 10.0 ** rng.uniform(-4, 6))
        target = thr * (1 + rng.choice([-1.0, 1.0]) * 10.0 ** -rng.uniform(3, 7)) if i % 4 else thr * rng.uniform(0.3, 1.2)
        lo, hi = 1e-9, 0.45
        for _ in range(40):
            mid = np.sqrt(lo * hi)
            r = tc._max_ratio_float(tc._interface_case(np.random.default_rng(i), ndim, d, mid, base, pert, scale), ndim,
                                    d, EPS)
            lo, hi = (mid, hi) if r < target else (lo, mid)
        out.append(tc._interface_case(np.random.default_rng(i), ndim, d, lo, base, pert, scale))
    return out


@pytest.mark.parametrize("ndim,d", [(1, 0), (2, 0), (2, 1), (3, 0), (3, 2)])
def test_mask_is_sound(lib, ndim, d):
    thr, thr_f, eps4_f = tc.scheme_thresholds()
    cases = _cases(ndim, d, thr)
    U, un, pn = (np.ascontiguousarray([c[k] for c in cases], dtype=np.float64) for k in range(3))
    alpha = np.array([c[7] for c in cases])
    a = np.ascontiguousarray(alpha[:, [0, 1, -1]])
    s = np.sqrt(U[:, 2:4, 0])
    sh = (U[:, 2:4, -1] + 2 * pn[:, 2:4]) / s
    su = U[:, 2:4, 1:-1] / s[..., None]
    args = [np.ascontiguousarray(x) for x in (U, un, pn, s, sh, su, a)]
    proven = 0
    for ulps in (-2, -1, 0, 1, 2):
        lib.closed_seed_ulps(ulps)
        out, _, _ = th.run(lib, ndim, d, args, float(thr_f), float(eps4_f))
        lib.closed_seed_ulps(0)
        for i in np.flatnonzero(out[:, 0]):
            u, hb1, hb2, hic = _exact_roe(s[i], sh[i], su[i], ndim)
            recs = tc._split_values_exact(U[i], un[i], pn[i], u, hb1, hb2, hic, alpha[i], ndim, d)
            mask = int(out[i, 2])
            for b, x in enumerate(recs):
                if (mask >> b) & 1:
                    continue
                proven += 1
                assert tc.exact_keep(x, thr_f, EPS), (ndim, d, i, b, ulps)
    assert proven > 100


def test_pairs_equal_singles():
    lib = _compile("cert_pairs_host.cpp")
    thr, thr_f, eps4_f = tc.scheme_thresholds()
    rng = np.random.default_rng(8)
    V = tc._value_cases(rng, thr, EPS, 4000).astype(np.float32)
    V = np.concatenate([V, rng.standard_normal((4000, 5)).astype(np.float32) *
                        10.0 ** rng.uniform(-30, 30, (4000, 1)).astype(np.float32)])
    V[::997, 2] = np.inf
    V[1::997, 3] = np.nan
    V = V[rng.permutation(len(V))]
    V = np.ascontiguousarray(V[: len(V) // 2 * 2].reshape(-1, 2, 5))
    d = (np.nanmax(np.abs(V), -1) * np.float32(32 * 2.0**-24) + np.float32(2.0**-90)).astype(np.float32)
    out = np.zeros((len(V), 2), dtype=np.int32)
    p = lambda x: x.ctypes.data_as(ctypes.c_void_p)
    lib.cert_pairs(ctypes.c_int64(len(V)), p(V), p(d), ctypes.c_float(float(thr_f)), ctypes.c_float(float(eps4_f)), p(out))
    assert np.array_equal(out[:, 0], out[:, 1])
    assert {0, 1, 2, 3} == set(out[:, 0].tolist())
