"""Paths that a rule on sizes or ranges selects, against the paths they stand
in for.

* one-launch 1D steps (teno_small.cu) against the staged entry points, which
  always take a launch per pass: the arithmetic is the same, so bit for bit;
  sizes at the edges of CTAs (127 cells), tiles (383), the cluster (16 CTAs) and
  the rule's limit (6144), every boundary type, body force, schemes;
* the wave speeds with cells skipped below the running maxima: the maxima of
  the same cells in another order, bit for bit;
* states inside and outside the range of the closed form's two-binary32 terms:
  the flux without flags against the flag path's (all binary64) at the parity
  tests' 1e-13."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2003_09145_gb300 import inputs  # noqa: E402
from parity import flux_scale, rel_max_err  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2003_09145_gb300 import api as A
    return A


def _line(n, seed):
    """A tube: smooth parts, jumps and noise; rho, p > 0."""
    rng = np.random.default_rng(seed)
    x = np.arange(n) / n
    rho = 1.0 + 0.3 * np.sin(7.0 * x + seed) + 0.5 * (x > 0.37) + 1e-3 * rng.standard_normal(n)
    p = 1.0 + 0.2 * np.cos(5.0 * x) + 2.0 * (x > 0.71)
    u = 0.4 * np.sin(3.0 * x) + 0.3 * (x > 0.55)
    return np.ascontiguousarray(inputs.prim_to_cons(rho, [u], p))


@pytest.mark.parametrize("n", [1, 2, 5, 31, 127, 128, 255, 1000, 2032, 2033, 6128, 6143, 6144, 6145])
@pytest.mark.parametrize("bc", [0, 1, 2, 3])
def test_small_step_equals_staged_step(api, n, bc):
    U0 = torch.from_numpy(_line(n, n + bc)).cuda()
    face = [[[1.2, 0.1, 2.9], [0.9, -0.2, 2.4]]] if bc == 3 else None
    grav = (0.3,) if n % 2 else None
    scheme = api.Scheme(scheme=["lad", "teno5", "teno5a"][n % 3])
    grid = api.EulerGrid((n,), (1.0 / n,), (bc,), scheme, grav, face)
    for dt_fixed, t_end in ((0.0, float("inf")), (1e-4 / n, float("inf")), (0.0, 1e-6 / n)):
        S = api.Solver(grid)
        U = U0.clone()
        S.step(U, t_end, dt_fixed)
        E = api.SlabEngine(grid)
        U1, U2, V = torch.empty_like(U0), torch.empty_like(U0), U0.clone()
        for k, (a, b) in enumerate(((U0, U1), (U1, U2), (U2, V)), start=1):
            E.begin(a)
            E.end(k, a, U0, b, t_end, dt_fixed)
        assert torch.equal(U, V)
        assert torch.equal(S.t, E.t) and torch.equal(S.dt, E.dt)
        assert S.status() == E.status() == 0


@pytest.mark.parametrize("n", [(200, 1), (1, 200), (6144, 1), (1, 1), (200, 1, 1), (1, 200, 1), (1, 1, 200), (3, 1, 40)])
@pytest.mark.parametrize("bc", [0, 1, 2])
def test_one_cell_across_equals_staged_step(api, n, bc):
    """2D and 3D grids of one cell across are no 1D grids: every momentum counts."""
    ndim = len(n)
    U = inputs.random_discontinuous_state(ndim, n, seed=sum(n))
    U[2:-1] += 0.3 * U[0]
    U[-1] += 0.5 * (U[1:-1] ** 2).sum(0) / U[0]
    U0 = torch.from_numpy(np.ascontiguousarray(U)).cuda()
    grid = api.EulerGrid(n, (0.01,) * ndim, (bc,) * ndim)
    S, E = api.Solver(grid), api.SlabEngine(grid)
    U, U1, U2, V = U0.clone(), torch.empty_like(U0), torch.empty_like(U0), U0.clone()
    S.step(U)
    for k, (a, b) in enumerate(((U0, U1), (U1, U2), (U2, V)), start=1):
        E.begin(a)
        E.end(k, a, U0, b, float("inf"), 0.0)
    assert torch.equal(U, V) and torch.equal(S.dt, E.dt)
    assert S.status() == E.status() == 0


def test_small_step_past_t_end_and_nonphysical(api):
    n = 300
    U0 = torch.from_numpy(_line(n, 3)).cuda()
    grid = api.EulerGrid((n,), (1.0 / n,), (1,))
    S = api.Solver(grid)
    S.reset_time(2.0)
    U = U0.clone()
    S.step(U, 1.0)
    assert torch.equal(U, U0) and S.dt.item() == 0.0 and S.t.item() == 2.0 and S.status() == 0
    U[0, 17] = -1.0
    S.reset_time(0.0)
    S.step(U)
    assert S.status() != 0


@pytest.mark.parametrize("ndim,n", [(1, (300000,)), (2, (601, 503)), (3, (97, 61, 53))])
@pytest.mark.parametrize("scale", [1.0, 2.0**-70, 2.0**65])
def test_speed_maxima_do_not_depend_on_the_order_of_cells(api, ndim, n, scale):
    U = inputs.random_discontinuous_state(ndim, n, seed=ndim) * scale
    if ndim > 1:
        U[-1] -= 0.5 * U[2] ** 2 / U[0]
        U[2] = 0.0                               # one direction at rest
    U = torch.from_numpy(np.ascontiguousarray(U)).cuda().reshape(ndim + 2, -1)
    E = api.SlabEngine(api.EulerGrid(n, (1.0,) * ndim, (0,) * ndim))
    words = []
    for V in (U, U.flip(1), U.roll(12345, 1), U[:, torch.argsort(U[0])], U[:, torch.argsort(U[-1] / U[0])]):
        E.begin(V.contiguous())
        words.append(E.alpha_words().clone())
    assert words[0][: 3 * ndim].min() >= 0 and words[0][0] > 0
    for w in words[1:]:
        assert torch.equal(w, words[0])


@pytest.mark.parametrize("ndim,n", [(1, (500,)), (2, (61, 47)), (3, (23, 19, 17))])
@pytest.mark.parametrize("krho,ku", [(0, 0), (-22, 0), (29, 0), (33, 0), (0, -18), (0, -21), (0, 31), (-40, 25), (12, 4)])
def test_closed_form_in_and_out_of_range(api, ndim, n, krho, ku):
    """rho scaled by 2^krho, velocities by 2^ku, pressure by 2^(krho + 2 ku)."""
    U = inputs.random_smooth_state(ndim, n, seed=5, amp=0.05)
    U[0] *= 2.0**krho
    U[1:-1] *= 2.0 ** (krho + ku)
    U[-1] *= 2.0 ** (krho + 2 * ku)
    dx = tuple(1.0 / m for m in n)
    # eps scaled with the split values (rho u), squared, so that the selections
    # are the unscaled state's
    s = api.Scheme(eps=1e-6 * 4.0 ** (krho + ku))
    grid = api.EulerGrid(n, dx, (0,) * ndim, s)
    Ut = torch.from_numpy(np.ascontiguousarray(U)).cuda()
    a, _ = api.rhs(grid, Ut, want_flags=True)
    b = api.rhs(grid, Ut)
    assert torch.isfinite(b).all()
    assert rel_max_err(b.cpu().numpy(), a.cpu().numpy(), flux_scale(U, n, dx)) <= 1e-13


@pytest.mark.parametrize("ndim", [2, 3])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("p0", [1.0, 1e5, 1e9])
def test_a_direction_at_rest_stays_at_rest(api, ndim, axis, p0):
    """A rough wave along one axis, uniform along the others: their momenta get exact zeros."""
    if axis >= ndim:
        pytest.skip("axis")
    rng = np.random.default_rng(axis)
    n = tuple(96 if k == axis else 7 for k in range(ndim))
    x = np.arange(96) / 96
    shape = tuple(96 if ndim - 1 - k == axis else 1 for k in range(ndim))
    wave = (np.sin(2.0 * np.pi * x) + 0.2 * rng.uniform(-1, 1, 96)).reshape(shape)
    full = tuple(reversed(n))
    rho = np.broadcast_to(1.0 + 0.01 * wave, full)
    vel = [np.broadcast_to((0.3 + 0.01 * wave) * np.sqrt(p0) if k == axis else 0.0 * wave, full) for k in range(ndim)]
    p = np.broadcast_to(p0 * (1.0 + 0.01 * wave), full)
    U = torch.from_numpy(np.ascontiguousarray(inputs.prim_to_cons(rho, vel, p))).cuda()
    grid = api.EulerGrid(n, (0.1,) * ndim, (0,) * ndim)
    R = api.rhs(grid, U)
    assert torch.isfinite(R).all() and R[1 + axis].abs().max() > 0
    for k in range(ndim):
        if k != axis:
            assert torch.count_nonzero(R[1 + k]).item() == 0


@pytest.mark.parametrize("ndim,n", [(1, (500,)), (2, (61, 47)), (3, (23, 19, 17))])
@pytest.mark.parametrize("krho,ku", [(-19, -18), (-10, -18), (-15, -15), (-20, -19), (-18, -10), (28, -18)])
def test_closed_form_with_both_scales_moved(api, ndim, n, krho, ku):
    """As above: the energy flux goes with rho u^3."""
    test_closed_form_in_and_out_of_range(api, ndim, n, krho, ku)


@pytest.mark.parametrize("ndim,n", [(1, (512,)), (2, (64, 40)), (3, (48, 16, 12))])
@pytest.mark.parametrize("p_cold", [1e-2, 1e-4, 1e-6, 1e-10, 1e-14, 1e-18, 1e-22, 1e-26, 1e-30])
def test_cold_region_beside_a_fast_one(api, ndim, n, p_cold):
    """The speeds are set by the fast half; in the cold one 1/c multiplies the corrections."""
    rng = np.random.default_rng(3)
    full = tuple(reversed(n))
    x = np.broadcast_to(np.arange(n[0]) / n[0], full)
    cold = (x > 0.25) & (x < 0.85)
    f = [1.0 + 0.02 * np.sin(2 * np.pi * (5 * x + rng.uniform())) + 0.01 * rng.uniform(-1, 1, full) for _ in range(3)]
    rho = f[0]
    p = np.where(cold, p_cold, 1.0) * f[1]
    vel = [np.where(cold, np.sqrt(p_cold) * 0.01 * rng.uniform(-1, 1, full), 0.7 * f[2]) for _ in range(ndim)]
    U = inputs.prim_to_cons(rho, vel, p)
    grid = api.EulerGrid(n, (1.0,) * ndim, (0,) * ndim)
    Ut = torch.from_numpy(np.ascontiguousarray(U)).cuda()
    a, _ = api.rhs(grid, Ut, want_flags=True)
    b = api.rhs(grid, Ut)
    assert torch.isfinite(b).all()
    assert rel_max_err(b.cpu().numpy(), a.cpu().numpy(), flux_scale(U, n, (1.0,) * ndim)) <= 1e-13


def _launches(api, grid, U):
    import ctypes
    lib, S = grid.lib, api.Solver(grid)
    ms, n = (ctypes.c_double * 4)(), (ctypes.c_int64 * 4)()
    lib.teno_timer_begin()
    S.step(U.clone())
    torch.cuda.synchronize()
    lib.teno_timer_end(ms, n)
    return sum(n)


@pytest.mark.parametrize("n", [1, 127, 128, 1016, 1017, 2032, 6144])
@pytest.mark.parametrize("bc", [0, 2, 3])
def test_small_steps_are_one_launch(api, n, bc):
    """The comparison above is of two paths: up to the rule's limit one launch, then several."""
    face = [[[1.2, 0.1, 2.9], [0.9, -0.2, 2.4]]] if bc == 3 else None
    U = torch.from_numpy(_line(n, 5)).cuda()
    assert _launches(api, api.EulerGrid((n,), (1.0 / n,), (bc,), None, None, face), U) == 1
    U = torch.from_numpy(_line(6145, 5)).cuda()
    assert _launches(api, api.EulerGrid((6145,), (1.0,), (bc,), None, None, face), U) >= 12
    U = torch.from_numpy(_line(n, 5)).cuda()
    assert _launches(api, api.EulerGrid((n,), (1.0 / n,), (bc,), api.Scheme(scheme="wenoz"), None, face), U) >= 9
