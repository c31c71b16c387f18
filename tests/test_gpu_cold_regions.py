"""Cold regions beside hot or fast ones, against extended precision.

The speeds are set by the hot part; in the cold one the characteristic rows go with
1/c, so terms that cancel in the flux exceed it by alpha / c.  Each flux may be off by
some 2^-50 of its flux scale (a few roundings of terms of that size), so a
right-hand side by 2 ndim of those, doubled for the primitives: 2e-14 covers three
directions, times the digits that the pressure loses in E (E (gamma - 1) / p, at
most 10 here: velocities of the order of the local sound speed)."""
import numpy as np
import pytest

import highprec
from paper_2003_09145_gb300 import inputs
from parity import flux_scale

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2003_09145_gb300 import api as A
    return A


@pytest.mark.parametrize("ndim,n", [(1, (60,)), (2, (14, 9)), (3, (9, 6, 5))])
@pytest.mark.parametrize("ratio", [1.0, 1e-2, 1e-4, 1e-6, 1e-8, 1e-10])
@pytest.mark.parametrize("scheme", ["lad", "teno5", "teno5a"])
@pytest.mark.parametrize("moving", [0.0, 0.7])
def test_cold_beside_hot(api, ndim, n, ratio, scheme, moving):
    worst = 0.0
    for seed in range(4):
        rng = np.random.default_rng(seed)
        full = tuple(reversed(n))
        x = np.broadcast_to(np.arange(n[0]) / n[0], full)
        cold = (x > 0.3) & (x < 0.8)
        amp = 10.0 ** rng.uniform(-3, -0.7)
        f = [1.0 + amp * rng.uniform(-1, 1, full) for _ in range(2 + ndim)]
        rho = f[0] * np.where(cold, 10.0 ** rng.uniform(-1, 1), 1.0)
        p = np.where(cold, ratio, 1.0) * f[1]
        vel = [np.where(cold, 0.3 * np.sqrt(ratio) * (f[2 + k] - 1.0) / amp, moving * f[2 + k]) for k in range(ndim)]
        U = np.ascontiguousarray(inputs.prim_to_cons(rho, vel, p))
        bc, dx = (seed % 3,) * ndim, (1.0,) * ndim
        grid = api.EulerGrid(n, dx, bc, api.Scheme(scheme=scheme, eps=(1e-6, 1e-2)[seed % 2]))
        Ut = torch.from_numpy(U).cuda()
        a, flags = api.rhs(grid, Ut, want_flags=True)
        want = highprec.rhs(U, n, dx, bc, flags.cpu().numpy() & 7).reshape(ndim + 2, -1)
        scale = flux_scale(U, n, dx).reshape(-1)[:ndim + 2]
        for R in (a, api.rhs(grid, Ut)):
            err = np.abs(R.cpu().numpy().reshape(ndim + 2, -1) - want).max(1) / scale
            worst = max(worst, float(err.max()))
    assert worst <= 2e-14


@pytest.mark.parametrize("ndim,n", [(1, (7,)), (1, (40,)), (2, (5, 32)), (2, (12, 9)), (3, (5, 6, 6))])
@pytest.mark.parametrize("gamma", [1.01, 1.1, 1.4, 3.0])
@pytest.mark.parametrize("scheme", ["lad", "teno5a"])
def test_slow_cold_beside_hot(api, ndim, n, gamma, scheme):
    """The cuts take out what the all-kept flux has of the hot side, larger than it by alpha / c."""
    cases = 0
    for seed in range(24):
        rng = np.random.default_rng(seed)
        full = tuple(reversed(n))
        x = np.broadcast_to(np.arange(n[0]) / n[0], full)
        cold = x > 0.5
        amp, ratio = 10.0 ** rng.uniform(-6, -1), 10.0 ** rng.uniform(-7, -3)

        def ripple():
            return 1.0 + amp * rng.uniform(-1, 1, full)

        rho, p = ripple(), np.where(cold, ratio, 1.0) * ripple()
        slow = np.sqrt(gamma * ratio) * rng.uniform(0.2, 2.0)
        vel = [np.where(cold, slow, 100.0 * slow) * rng.choice([-1, 1]) * rng.uniform(0.3, 1) * ripple()
               for _ in range(ndim)]
        U = np.ascontiguousarray(np.stack([rho] + [rho * v for v in vel] +
                                          [p / (gamma - 1) + 0.5 * rho * sum(v * v for v in vel)]))
        cond = float((U[-1] * (gamma - 1) / p).max())
        if cond > 10.0:
            continue
        bc, dx = tuple((0, 1, 2)[(seed + k) % 3] for k in range(ndim)), (1.0,) * ndim
        s = api.Scheme(scheme=scheme, gamma=gamma, eps=(1e-6, 1e-2)[seed % 2], b_l=(4, 1)[seed % 2], b_u=(10, 2)[seed % 2])
        grid = api.EulerGrid(n, dx, bc, s)
        Ut = torch.from_numpy(U).cuda()
        a, flags = api.rhs(grid, Ut, want_flags=True)
        sel = flags.cpu().numpy() & 7
        want = highprec.rhs(U, n, dx, bc, sel, gamma).reshape(ndim + 2, -1)
        scale = flux_scale(U, n, dx, gamma).reshape(-1)[:ndim + 2]
        # Where a selected candidate holds the jump (a cold region of two cells has no other), the
        # answer itself is that sensitive: one rounding of U moves the exact right-hand side by up
        # to 1e-11 of the flux scale.  Well conditioned: by less than a tenth of the bound.
        nudged = highprec.rhs(U * (1 + 2.0**-52 * rng.choice([-1, 0, 1], U.shape)), n, dx, bc, sel, gamma)
        if (np.abs(nudged.reshape(ndim + 2, -1) - want).max(1) / scale).max() > 2e-15:
            continue
        cases += 1
        for R in (a, api.rhs(grid, Ut)):
            err = np.abs(R.cpu().numpy().reshape(ndim + 2, -1) - want).max(1) / scale
            assert err.max() <= 2e-14 * cond, (seed, cond, float(err.max()))
    assert cases >= 3
