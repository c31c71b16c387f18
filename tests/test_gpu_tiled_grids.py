"""Grids of one size class against the same cells on a grid of another, bit for bit.

A grid tiled from a small one (repeated along periodic axes; along walls a tile
that ends in its own mirror image, so that a tile's neighbour is its wall's ghost)
has the small grid's speeds and, in every tile, its right-hand side: the
arithmetic of an interface does not depend on where it lies.  So does a step, but
where tiles meet along a walled axis (a stage's state need not be mirrored to the
last bit).  The classes take
different kernels: up to 2^17 cells one closed-form launch for all directions, up to
2^25 a flux buffer and list per direction with one correction and one difference
launch, beyond that one direction after another, and beyond 3 2^27 without binary32
planes of the cells."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2003_09145_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu
PERIODIC, TRANSMISSIVE, REFLECTIVE, DIRICHLET = 0, 1, 2, 3


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2003_09145_gb300 import api as A
    return A


def _tile_state(n, bc, seed):
    """Blocks and noise on n cells; along a walled axis the second half mirrors the first."""
    ndim = len(n)
    half = tuple(m // 2 if b == REFLECTIVE else m for m, b in zip(n, bc))
    U = inputs.random_discontinuous_state(ndim, half, seed=seed)
    U[1:-1] += 0.2 * U[0]
    U[-1] += 0.5 * (U[1:-1] ** 2).sum(0) / U[0]
    for d in range(ndim):
        if bc[d] == REFLECTIVE:
            ax = ndim - d
            V = np.flip(U, ax).copy()
            V[1 + d] *= -1.0
            U = np.concatenate([U, V], axis=ax)
    return np.ascontiguousarray(U)


def _need(nbytes):
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    if free < nbytes:
        pytest.skip(f"needs {nbytes / 2**30:.0f} GiB of free device memory, {free / 2**30:.0f} GiB free")


def _same_in_every_tile(big, small, n, reps):
    """big [nvar][..][reps n].. equals small in every tile (axes slowest first), slice by slice."""
    ndim = len(n)
    shape = [small.shape[0]]
    one = [small.shape[0]]
    for d in reversed(range(ndim)):
        shape += [reps[d], n[d]]
        one += [1, n[d]]
    for v in range(small.shape[0]):
        if not torch.equal(big.reshape(shape)[v], small.reshape(one)[v].expand(shape[1:])):
            return False
    return True


CASES = [
    # tile, boundaries, gravity, repetitions of each larger grid
    ((96,), (PERIODIC,), None, [(73,), (350003,), (4194400,)]),
    ((40, 30), (PERIODIC, REFLECTIVE), (0.1, -0.2), [(8, 28), (170, 170), (480, 700), (224, 1), (28100, 1)]),
    ((36, 52), (REFLECTIVE, DIRICHLET), (0.0, 0.3), [(80, 1), (18000, 1), (216000, 1)]),
    ((64, 46), (TRANSMISSIVE, PERIODIC), None, [(1, 60), (1, 11500)]),
    ((16, 12, 10), (PERIODIC, PERIODIC, PERIODIC), None, [(5, 4, 4), (28, 26, 25), (64, 55, 60)]),
    ((20, 14, 18), (REFLECTIVE, PERIODIC, DIRICHLET), (0.1, 0.0, -0.3), [(6, 5, 1), (80, 90, 1), (1, 32, 1), (1, 6800, 1)]),
    ((12, 10, 16), (DIRICHLET, REFLECTIVE, TRANSMISSIVE), (0.1, 0.2, 0.3), [(1, 90, 1)]),
]


@pytest.mark.parametrize("case,k", [(c, k) for c in range(len(CASES)) for k in range(len(CASES[c][3]))])
def test_tiles_equal_the_small_grid(api, case, k):
    n, bc, grav, sizes = CASES[case]
    reps = sizes[k]
    ndim = len(n)
    U0 = _tile_state(n, bc, seed=case)
    p0 = inputs.prim_to_cons(np.array([0.8]), [np.array([0.1 * (d + 1)]) for d in range(ndim)], np.array([1.1]))[:, 0]
    faces = [[list(p0), list(1.2 * p0)] if b == DIRICHLET else None for b in bc] if DIRICHLET in bc else None
    dx = tuple(0.02 + 0.01 * d for d in range(ndim))
    small = api.EulerGrid(n, dx, bc, None, grav, faces)
    big = api.EulerGrid(tuple(m * r for m, r in zip(n, reps)), dx, bc, None, grav, faces)
    S0 = torch.from_numpy(U0).cuda()
    rep = (1,) + tuple(reversed(reps))
    _need(int(1.05 * (3 * 8 * (ndim + 2) * big.ncell + big.workspace_bytes(1))))
    R0 = api.rhs(small, S0)
    B = S0.repeat(rep)
    R = api.rhs(big, B)
    assert torch.isfinite(R0).all() and R0.abs().max() > 0
    assert _same_in_every_tile(R, R0, n, reps)
    del R
    torch.cuda.empty_cache()
    if any(b == REFLECTIVE and r > 1 for b, r in zip(bc, reps)):
        return
    # one step in stages on the small grid (its own small path aside), a plain one on the big
    E, S = api.SlabEngine(small), api.Solver(big)
    U1, U2, V = torch.empty_like(S0), torch.empty_like(S0), S0.clone()
    for s, (a, b) in enumerate(((S0, U1), (U1, U2), (U2, V)), start=1):
        E.begin(a)
        E.end(s, a, S0, b)
    S.step(B)
    assert torch.equal(S.dt, E.dt) and S.status() == E.status() == 0
    assert _same_in_every_tile(B, V, n, reps)
    del B, S
    torch.cuda.empty_cache()


def test_tiles_beyond_the_fixed_points_range(api):
    """Fluxes that the closed form leaves unwritten (values above 2^1007), on a list of indices."""
    n, reps = (96,), (4194400,)
    U0 = torch.from_numpy(_tile_state(n, (PERIODIC,), seed=1) * 2.0**1012).cuda()
    small = api.EulerGrid(n, (1.0,), (PERIODIC,))
    big = api.EulerGrid((n[0] * reps[0],), (1.0,), (PERIODIC,))
    _need(int(1.05 * (2 * 24 * big.ncell + big.workspace_bytes(0))))
    R0 = api.rhs(small, U0)
    assert torch.isfinite(R0).all() and R0.abs().max() > 2.0**1000
    assert _same_in_every_tile(api.rhs(big, U0.repeat((1, reps[0]))), R0, n, reps)
