"""The paper's comparison schemes on the GPU (teno_grid.scheme): TENO5 with a
fixed C_T = 1e-7 (Sec. 2, Sec. 4), TENO5-A (eq. 2.16-2.18) and WENO-Z
(tau_5 of eq. 2.12), through the same C-ABI entry points, against the oracle
run with the same scheme.

Tolerances as for the LAD path: 1e-12 relative max-norm on one RHS (flag
path and the benchmark's flag-free path), selections identical except
counted rounding-boundary flips, 1e-10 relative L1 after a run of steps."""
import numpy as np
import pytest

from paper_2003_09145_gb300 import inputs
from parity import RHS_RTOL, STEP_RTOL, compare_rhs, flux_scale, rel_l1_err, rel_max_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SCHEMES = ["teno5", "teno5a", "wenoz"]


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2003_09145_gb300 import api as A
    return A


def _problems():
    return {
        "sod": inputs.shock_tube(200),
        "shu": inputs.shu_osher(4096),
        "rand2d": inputs.Problem("r2", inputs.random_discontinuous_state(2, (40, 30), seed=5), (40, 30),
                                 (0.02, 0.03), (1, 0), 0.0),
        "rand3d": inputs.Problem("r3", inputs.random_discontinuous_state(3, (12, 10, 9), seed=6), (12, 10, 9),
                                 (0.1, 0.1, 0.1), (0, 1, 0), 0.0),
        "quad128": inputs.riemann_2d(n=128),
        "turb32": inputs.solenoidal_turbulence(n=32),
    }


@pytest.mark.parametrize("scheme", SCHEMES)
@pytest.mark.parametrize("case", ["sod", "shu", "rand2d", "rand3d", "quad128", "turb32"])
def test_rhs_matches_oracle(api, oracle, scheme, case):
    P = _problems()[case]
    sch = api.Scheme(gamma=P.gamma, scheme=scheme, ct_m=7)
    params = oracle.Params(gamma=P.gamma, scheme=scheme, ct_m=7)
    grid = api.EulerGrid(P.n, P.dx, P.bc, sch)
    U = torch.from_numpy(np.ascontiguousarray(P.U0)).cuda()
    a, fl = api.rhs(grid, U, want_flags=True)
    b = api.rhs(grid, U, want_flags=False)
    torch.cuda.synchronize()
    a, fl, b = a.cpu().numpy(), fl.cpu().numpy(), b.cpu().numpy()
    fs = flux_scale(P.U0, P.n, P.dx, P.gamma)
    for R in (a, b):
        err, rep = compare_rhs(P.U0, P.n, P.dx, P.bc, R, fl, oracle, params)
        assert not rep.unexplained, rep.unexplained[:3]
        assert rep.mismatched <= rep.total * 1e-4
        assert err <= RHS_RTOL, err
    assert rel_max_err(b, a, fs) <= 1e-13
    m = fl >> 3
    if scheme == "teno5":
        assert np.all(m == 7)
    elif scheme == "teno5a":
        assert np.all((m >= 7) & (m <= 10))
    else:
        assert np.all(fl == 7)


@pytest.mark.parametrize("scheme", SCHEMES)
def test_sod_run_matches_oracle(api, oracle, scheme):
    P = inputs.shock_tube(200)
    grid = api.EulerGrid(P.n, P.dx, P.bc, api.Scheme(scheme=scheme))
    U = torch.from_numpy(P.U0.copy()).cuda()
    solver = api.Solver(grid, cfl=P.cfl)
    solver.run(U, P.t_end)
    torch.cuda.synchronize()
    Uo, to, ko = oracle.euler_run(P.U0, P.n, P.dx, P.bc, P.t_end, sigma=P.cfl,
                                  params=oracle.Params(scheme=scheme))
    assert abs(solver.t.item() - P.t_end) <= 1e-14
    assert rel_l1_err(U.cpu().numpy(), Uo) <= STEP_RTOL


@pytest.mark.parametrize("scheme", SCHEMES)
def test_scalar_mode_matches_oracle(api, oracle, scheme):
    n = 200
    dx = 2.0 / n
    for u0 in (inputs.scalar_smooth(n), inputs.scalar_composite(n)):
        adv = api.ScalarAdvection(n, dx, mode="lad", scheme=api.Scheme(scheme=scheme))
        r = adv.rhs(torch.from_numpy(u0).cuda()).cpu().numpy()
        ro = oracle.scalar_rhs(u0, dx, "lad", oracle.Params(scheme=scheme))
        assert np.max(np.abs(r - ro)) <= RHS_RTOL * np.max(np.abs(u0)) / dx


@pytest.mark.parametrize("scheme", ["teno5", "teno5a"])
def test_adjoint_of_teno_variants(api, oracle, scheme):
    """The TENO cutoffs are piecewise constant, so the adjoint (selections
    frozen) applies to every TENO variant."""
    from oracle import grad
    U = inputs.random_discontinuous_state(2, (19, 13), seed=3)
    n, dx, bc = (19, 13), (0.1, 0.08), (0, 1)
    rng = np.random.default_rng(7)
    Rbar = rng.standard_normal(U.shape)
    ref, _ = grad.rhs_vjp(U, n, dx, bc, Rbar, oracle.Params(scheme=scheme))
    grid = api.EulerGrid(n, dx, bc, api.Scheme(scheme=scheme))
    got = api.rhs_adjoint(grid, torch.from_numpy(U).cuda(), torch.from_numpy(Rbar).cuda()).cpu().numpy()
    assert np.max(np.abs(got - ref)) / np.max(np.abs(ref)) <= 1e-10


def test_wenoz_adjoint_unsupported(api):
    from paper_2003_09145_gb300 import _lib
    grid = api.EulerGrid((16,), (0.1,), (1,), api.Scheme(scheme="wenoz"))
    U = torch.from_numpy(inputs.shock_tube(16).U0).cuda()
    with pytest.raises(RuntimeError, match="UNSUPPORTED"):
        api.rhs_adjoint(grid, U, torch.ones_like(U))


def test_teno5_fixed_equals_lad_with_one_magnitude(api):
    """TENO5 at C_T = 1e-7 and LAD with B_l = 7, B_u = 8 keep the same
    stencils everywhere (m differs only where tau_5 = 0, where both keep all),
    so the flag paths (binary64 selections everywhere) agree bit for bit."""
    P = inputs.riemann_2d(n=96)
    U = torch.from_numpy(P.U0).cuda()
    a, fa = api.rhs(api.EulerGrid(P.n, P.dx, P.bc, api.Scheme(scheme="teno5", ct_m=7)), U, want_flags=True)
    b, fb = api.rhs(api.EulerGrid(P.n, P.dx, P.bc, api.Scheme(b_l=7, b_u=8)), U, want_flags=True)
    assert torch.equal(a, b)
    assert torch.equal(fa & 7, fb & 7)


@pytest.mark.parametrize("k", [-480, -300, -170, -146, -130, -60, 0, 60, 130, 143, 146, 150, 155, 170, 330, 480])
@pytest.mark.parametrize("fixed_eps", [False, True])
def test_wenoz_at_any_scale(api, k, fixed_eps):
    """WENO-Z is homogeneous in (u, sqrt(eps)): data times 2^k with eps times 4^k
    give 2^k times the right-hand side (the products of the weights round alike up
    to their range's ends; 1e-14 covers the divided weights beyond)."""
    rng = np.random.default_rng(4)
    n = 300
    u = np.sin(2 * np.pi * np.arange(n) / 40.0) + (np.arange(n) > 150) + 0.1 * rng.standard_normal(n)
    e0, ek = (1e-6 * 4.0**-k, 1e-6) if fixed_eps else (1e-6, 1e-6 * 4.0**k)
    R = []
    for s, eps in ((0, e0), (k, ek)):
        adv = api.ScalarAdvection(n, 1.0 / n, scheme=api.Scheme(scheme="wenoz", eps=eps))
        R.append(adv.rhs(torch.from_numpy(u * 2.0**s).cuda()).cpu().numpy())
    assert np.isfinite(R[1]).all()
    assert np.max(np.abs(R[1] * 2.0**-k - R[0])) <= 1e-14 * n * np.max(np.abs(u))


def _flux_from_flags(U, bc, flags, gamma=1.4):
    """The 1D fluxes with the selections of ``flags`` (the flag layout of teno.h),
    every step from the paper's equations; no stencil at all gives a field 0."""
    n = U.shape[1]
    i = np.arange(-3, n + 3)
    P = U[:, i % n if bc == 0 else np.clip(i, 0, n - 1)]
    rho, m, E = P
    u = m / rho
    p = (gamma - 1) * (E - 0.5 * rho * u * u)
    c = np.sqrt(gamma * p / rho)
    al = [np.abs(u - c).max(), np.abs(u).max(), np.abs(u + c).max()]
    F = np.array([m, m * u + p, u * (E + p)])
    a, b = slice(2, n + 3), slice(3, n + 4)
    sa, sb = np.sqrt(rho[a]), np.sqrt(rho[b])
    ut = (sa * u[a] + sb * u[b]) / (sa + sb)
    H = (sa * (E[a] + p[a]) / rho[a] + sb * (E[b] + p[b]) / rho[b]) / (sa + sb)
    c2 = (gamma - 1) * (H - 0.5 * ut * ut)
    cs, b1 = np.sqrt(c2), (gamma - 1) / c2

    def left(X):
        A = 0.5 * b1 * (0.5 * ut * ut * X[0] - ut * X[1] + X[2])
        B = 0.5 * (ut * X[0] - X[1]) / cs
        return [A + B, X[0] - 2 * A, A - B]

    def omega(sel):
        d = np.array([(sel >> k) & 1 for k in range(3)]) * np.array([0.1, 0.6, 0.3])[:, None]
        s = d.sum(0)
        return d / np.where(s > 0, s, 1.0)

    sel = flags.reshape(3, 2, n + 1) & 7
    W = [left(P[:, j:j + n + 1]) for j in range(6)]
    G = [left(F[:, j:j + n + 1]) for j in range(6)]
    f = []
    for s in range(3):
        tot = 0.0
        for side, sgn, order in ((0, 1.0, range(5)), (1, -1.0, range(5, 0, -1))):
            v = [0.5 * (G[j][s] + sgn * al[s] * W[j][s]) for j in order]
            o = omega(sel[s, side])
            tot = tot + (o[0] * (2 * v[0] - 7 * v[1] + 11 * v[2]) + o[1] * (-v[1] + 5 * v[2] + 2 * v[3]) +
                         o[2] * (2 * v[2] + 5 * v[3] - v[4])) / 6.0
        f.append(tot)
    mass = f[0] + f[1] + f[2]
    return np.array([mass, ut * mass + cs * (f[2] - f[0]),
                     f[0] * (H - ut * cs) + 0.5 * ut * ut * f[1] + f[2] * (H + ut * cs)]), sel


def test_selection_of_no_stencil(api):
    """B_l = 0 gives C_T = 1 at strong jumps, where no chi_k reaches it: the field
    contributes nothing, on the flag path and on the flag-free one (which the steps take) alike."""
    P = inputs.shock_tube(200)
    grid = api.EulerGrid(P.n, P.dx, P.bc, api.Scheme(b_l=0, b_u=4))
    U0 = P.U0 * (1.0 + 1e-3 * np.random.default_rng(1).standard_normal(P.U0.shape))
    U = torch.from_numpy(np.ascontiguousarray(U0)).cuda()
    a, flags = api.rhs(grid, U, want_flags=True)
    b = api.rhs(grid, U)
    F, sel = _flux_from_flags(U0, 1, flags.cpu().numpy())
    assert np.count_nonzero(sel == 0) >= 4
    want = (F[:, :-1] - F[:, 1:]) / P.dx[0]
    scale = flux_scale(U0, P.n, P.dx)
    assert rel_max_err(a.cpu().numpy(), want, scale) <= RHS_RTOL
    assert rel_max_err(b.cpu().numpy(), want, scale) <= RHS_RTOL
