"""Workspace sizes: the largest grids (more than 3 2^27 cells) and the adjoint hold no
more than the arrays listed here, so that a box which fills the card still fits --
primitives, half fluxes, one direction's interface fluxes, a list of interfaces, and
for a step the right-hand side and two stages."""
import ctypes

import pytest

from paper_2003_09145_gb300 import _lib


def _r(x):
    return (x + 255) // 256 * 256


def _faces(n):
    cells = 1
    for m in n:
        cells *= m
    return cells, max(cells // m * (m + 1) for m in n)


@pytest.mark.parametrize("n", [(3 * 2**27 + 1,), (2**31,), (20100, 20100), (65536, 65520), (739, 739, 739), (700, 900, 1100),
                               (929, 929, 929)])
@pytest.mark.parametrize("bc", [0, 2, 3])
def test_step_and_rhs(n, bc):
    lib, nd = _lib.load(), len(n)
    face = [[[1.0] + [0.0] * nd + [2.5] + [0.0] * (3 - nd)] * 2] * 3 if bc == 3 else None
    g = _lib.make_grid(n, (1.0,) * nd, (bc,) * nd, 1.4, 10.0, 4, 10, 1e-6, "lad", 7, None, face)
    N, M = _faces(n)
    nv, aux = nd + 2, 2 * nd + 3
    rhs = 256 + _r(8 * aux * N) + _r(8 * nd * (nv - 1) * N) + _r(8 * nv * M) + _r(4 * M) + \
        _r(8 * 6 * (nv + aux + nd * (nd + 1)))
    got = [lib.teno_workspace_bytes(ctypes.byref(g), op) for op in (0, 1)]
    slack = 8 * 6 * 2 * (nd + 2)                  # the ghost cells' binary32 values
    assert 0 < got[0] <= rhs + _r(slack)
    assert 0 < got[1] <= rhs + 3 * _r(8 * nv * N) + _r(slack)


@pytest.mark.parametrize("n", [(5000,), (10**8,), (300, 200), (12000, 10000), (32, 32, 32), (500, 500, 500)])
def test_adjoint(n):
    lib, nd = _lib.load(), len(n)
    g = _lib.make_grid(n, (1.0,) * nd, (0,) * nd, 1.4, 10.0, 4, 10, 1e-6, "lad", 7, None, None)
    N, M = _faces(n)
    nv, aux = nd + 2, 2 * nd + 3
    nsm = 152
    common = nd * (_r(24 * nv * M) + _r(48 * nv * M) + _r(M)) + 2 * _r(4 * (2 * M + 2)) + \
        _r(4 * (8 * nsm + 2)) + _r(8 * 6 * 8 * nsm * nd) + _r(8 * 18 * 8 * nsm)
    rhs = 1024 + _r(8 * aux * N) + common
    step = 1024 + 3 * _r(8 * aux * N) + common + _r(8 * nd * (nv - 1) * N) + 5 * _r(8 * nv * N) + \
        2 * _r(8 * nd * (nd + 8) * M)
    got = [lib.teno_adjoint_workspace_bytes(ctypes.byref(g), op) for op in (2, 3)]
    assert 0 < got[0] <= rhs and 0 < got[1] <= step
