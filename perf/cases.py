"""The calls that programs built on this framework make, over their real range
of sizes, for timing and for comparing results.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges,
``prepare`` makes what a program holds before the call (grid, solver with its
workspace, state), ``run`` is one pass through ``paper_2003_09145_gb300.api``,
``work`` what a pass cannot do without, ``exact`` the same result in plain
binary64 torch, written from the paper's equations without the library.

States are synthetic and seeded, shaped like the flows the solver advances
after their first steps: shocks and contacts smeared over one to three cells
between smooth regions, solenoidal turbulence with a few per cent of density
fluctuation, a perturbed heavy-over-light interface.  A step is timed on a
fresh copy of the same state (an in-place step would otherwise march through
other flows from pass to pass).
"""
import math

import torch

from paper_2003_09145_gb300 import api
from paper_2003_09145_gb300.inputs import PERIODIC, REFLECTIVE, TRANSMISSIVE

DIRICHLET = 3
EPS, H_LAD, B_L, B_U = 1e-6, 10.0, 4, 10


def listed():
    return [
        # the smallest call: one step of Sod's tube at the paper's kind of size
        # (a run takes a few hundred of them, so latency and launches count)
        {"name": "step1d_200", "call": "step", "flow": "tube", "n": "200", "bc": TRANSMISSIVE},
        # shock/entropy-wave interaction on 4096 cells, a few thousand steps a run
        {"name": "step1d_4096", "call": "step", "flow": "shu", "n": "4096", "bc": TRANSMISSIVE},
        # four-quadrant Riemann problem: a quick look, and the production size
        {"name": "step2d_512", "call": "step", "flow": "quad", "n": "512x512", "bc": TRANSMISSIVE},
        {"name": "step2d_2048", "call": "step", "flow": "quad", "n": "2048x2048", "bc": TRANSMISSIVE},
        # Rayleigh-Taylor: walls, fixed-state faces and the body force, ragged sizes
        {"name": "step2d_rt_129x515", "call": "step", "flow": "rt", "n": "129x515", "bc": REFLECTIVE},
        # the right-hand side alone on ragged transmissive 3D data (a user's own integrator)
        {"name": "rhs3d_97x61x45", "call": "rhs", "flow": "smooth", "n": "97x61x45", "bc": TRANSMISSIVE},
        # the comparison scheme without a cutoff: every face takes characteristic variables
        {"name": "rhs2d_wenoz_1024", "call": "rhs", "flow": "quad", "n": "1024x1024", "bc": TRANSMISSIVE,
         "scheme": "wenoz"},
        # turbulence in a periodic box: a coarse run and the production size
        {"name": "step3d_64", "call": "step", "flow": "turb", "n": "64x64x64", "bc": PERIODIC},
        {"name": "step3d_256", "call": "step", "flow": "turb", "n": "256x256x256", "bc": PERIODIC},
        # thousands of uneven shock tubes advanced together
        {"name": "batch_4096", "call": "batch", "nprob": 4096, "n_min": 64, "n_max": 4096},
        # the reverse of one step (gradients by checkpointing)
        {"name": "adjoint3d_128", "call": "adjoint", "flow": "turb", "n": "128x128x128", "bc": PERIODIC},
        # a whole differentiable rollout, forward and backward, as a training loop calls it
        {"name": "rollout3d_64", "call": "rollout", "flow": "turb", "n": "64x64x64", "bc": PERIODIC, "steps": 4},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step1d", "step1d", "step2d", "step2d", "rt", "rhs3d", "step3d", "step3d", "scheme", "batch",
                       "adjoint", "rollout"])
    if kind == "step1d":
        return {"call": "step", "flow": rng.choice(["tube", "shu"]), "n": str(size(64, 16384)),
                "bc": rng.choice([TRANSMISSIVE, TRANSMISSIVE, REFLECTIVE])}
    if kind == "step2d":
        return {"call": "step", "flow": "quad", "n": f"{size(64, 2048)}x{size(64, 2048)}", "bc": TRANSMISSIVE}
    if kind == "rt":
        return {"call": "step", "flow": "rt", "n": f"{size(32, 256)}x{size(128, 1024)}", "bc": REFLECTIVE}
    if kind == "rhs3d":
        return {"call": "rhs", "flow": "smooth", "n": f"{size(16, 200)}x{size(16, 200)}x{size(16, 200)}",
                "bc": rng.choice([TRANSMISSIVE, PERIODIC, REFLECTIVE])}
    if kind == "step3d":
        m = size(24, 224)
        return {"call": "step", "flow": "turb", "n": f"{m}x{m}x{m}", "bc": PERIODIC}
    if kind == "scheme":
        return {"call": "rhs", "flow": "quad", "n": f"{size(64, 1024)}x{size(64, 1024)}", "bc": TRANSMISSIVE,
                "scheme": rng.choice(["teno5", "teno5a", "wenoz"])}
    if kind == "batch":
        return {"call": "batch", "nprob": size(16, 4096), "n_min": 64, "n_max": size(256, 4096)}
    m = size(24, 112) if kind == "adjoint" else size(16, 64)
    c = {"call": kind, "flow": "turb", "n": f"{m}x{m}x{m}", "bc": PERIODIC}
    if kind == "rollout":
        c["steps"] = rng.choice([2, 4, 6])
    return c


# ---------------------------------------------------------------------------
# what a program holds
# ---------------------------------------------------------------------------
def _dims(case):
    return tuple(int(v) for v in case["n"].split("x"))


def _box(case):
    """Grid spacing, boundary types, gamma, body force and face states."""
    n = _dims(case)
    flow = case["flow"]
    if flow == "turb":
        return tuple(2.0 * math.pi / m for m in n), (case["bc"],) * len(n), 1.4, None, None
    if flow == "rt":
        g = 5.0 / 3.0
        faces = [None, [[2.0, 0.0, 0.0, 1.0 / (g - 1.0)], [1.0, 0.0, 0.0, 2.5 / (g - 1.0)]]]
        return (0.25 / n[0], 1.0 / n[1]), (REFLECTIVE, DIRICHLET), g, (0.0, 1.0), faces
    length = 10.0 if flow == "shu" else 1.0
    return tuple(length / m for m in n), (case["bc"],) * len(n), 1.4, None, None


def _cons(rho, vel, p, gamma):
    q2 = sum(v * v for v in vel)
    return torch.stack([rho] + [rho * v for v in vel] + [p / (gamma - 1.0) + 0.5 * rho * q2]).contiguous()


def _front(x, x0, width):
    return 0.5 * (1.0 + torch.tanh((x - x0) / width))


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _centres(n):
    """Cell-centre coordinates in [0, 1] per direction, shaped to broadcast over [n_z][n_y][n_x]."""
    out = []
    for d, m in enumerate(n):
        x = (torch.arange(m, device="cuda", dtype=torch.float64) + 0.5) / m
        out.append(x.reshape([m if k == len(n) - 1 - d else 1 for k in range(len(n))]))
    return out


def _state(case, seed):
    n = _dims(case)
    g = torch.Generator(device="cuda").manual_seed(1000003 * (seed + 1) + 7)
    shape = tuple(reversed(n))
    flow = case["flow"]
    gamma = _box(case)[2]
    x = _centres(n)
    if flow == "tube":
        # rarefaction, contact and shock between Sod-like states
        r = _rand(g, 6)
        h = 1.0 / n[0]
        fan, con, sho = _front(x[0], 0.35 + 0.05 * r[0], 0.04), _front(x[0], 0.55 + 0.05 * r[1], 2.0 * h), \
            _front(x[0], 0.75 + 0.05 * r[2], 0.8 * h)
        rho = 1.0 + 0.2 * r[3] - (0.55 * fan + 0.17 * con + 0.14 * sho) * (1.0 + 0.2 * r[3])
        p = (1.0 + 0.2 * r[4]) * (1.0 - 0.69 * fan - 0.2 * sho)
        u = 0.92 * fan - 0.9 * sho
        return _cons(rho, [u], p, gamma)
    if flow == "shu":
        # a strong shock running into a density wave, compressed waves behind it
        r = _rand(g, 4)
        s = 1.0 - _front(x[0], 0.3 + 0.2 * r[0], 0.8 / n[0])
        wave = torch.sin(50.0 * (x[0] + r[1]))
        rho = s * (3.857143 + 0.6 * torch.sin(170.0 * (x[0] + r[2]))) + (1.0 - s) * (1.0 + 0.2 * wave)
        u = s * (2.629369 + 0.1 * torch.sin(60.0 * (x[0] + r[3])))
        p = s * (10.3333 + 0.5 * torch.sin(60.0 * (x[0] + r[3]))) + (1.0 - s)
        return _cons(rho, [u], p, gamma)
    if flow == "quad":
        # curved shocks and slip lines of a four-quadrant problem with smooth flow between
        r = _rand(g, 12)
        X, Y = x[0], x[1]
        w = 1.2 / max(n)
        a = _front(X + 0.05 * torch.sin(5.0 * Y + 6.0 * r[0]), 0.6 + 0.2 * r[1], w)
        b = _front(Y + 0.05 * torch.sin(5.0 * X + 6.0 * r[2]), 0.6 + 0.2 * r[3], w)
        ne, nw, sw, se = a * b, (1.0 - a) * b, (1.0 - a) * (1.0 - b), a * (1.0 - b)

        def wave(k, q):
            return 1.0 + 0.03 * torch.sin(k * math.pi * (X + 0.7 * Y + q)) * torch.sin(k * math.pi * (Y - 0.6 * X + q))

        rho = (1.5 * ne + 0.5323 * (nw + se) + 0.138 * sw) * wave(6.0, r[4])
        u = 1.206 * (nw + sw) * wave(4.0, r[5])
        v = 1.206 * (se + sw) * wave(4.0, r[6])
        p = (1.5 * ne + 0.3 * (nw + se) + 0.029 * sw) * wave(5.0, r[7])
        return _cons(rho, [u, v], p, gamma)
    if flow == "rt":
        r = _rand(g, 6)
        X, Y = 0.25 * x[0], x[1]
        top = _front(Y + 0.02 * torch.cos(8.0 * math.pi * X) + 0.004 * torch.cos(24.0 * math.pi * X + 6.0 * r[0]), 0.5,
                     1.2 / n[1])
        rho = 2.0 - top
        p = (2.0 * Y + 1.0) * (1.0 - top) + (Y + 1.5) * top
        c = torch.sqrt(gamma * p / rho)
        decay = torch.exp(-20.0 * (Y - 0.5) ** 2)
        v = -0.05 * c * decay * torch.cos(8.0 * math.pi * X) * (1.0 + 0.3 * r[1])
        u = 0.03 * c * decay * torch.sin(8.0 * math.pi * X) * (1.0 + 0.3 * r[2])
        return _cons(rho.expand(shape), [u.expand(shape), v.expand(shape)], p.expand(shape), gamma)
    if flow == "smooth":
        r = _rand(g, 5, len(n) + 1)

        def field(i):
            arg = sum((1.0 + (i + k) % 3) * 2.0 * math.pi * xi + 6.0 * r[i][k]
                      for k, xi in enumerate(x))
            return torch.sin(arg + 6.0 * r[i][-1])

        vel = [0.4 * field(k) for k in range(len(n))]
        return _cons((1.0 + 0.25 * field(3)).expand(shape), [v.expand(shape) for v in vel],
                     (1.0 + 0.2 * field(4)).expand(shape), gamma)
    # turbulence: random-phase solenoidal velocity, E(k) ~ k^4 exp(-2 (k/4)^2), Mach 0.6, c = 1,
    # with a few per cent of isentropic density fluctuation
    ks = [torch.fft.fftfreq(m, d=1.0 / m, device="cuda", dtype=torch.float64).reshape(
        [m if k == a else 1 for k in range(3)]) for a, m in enumerate(shape)]
    K2 = sum(k * k for k in ks)
    K = torch.sqrt(K2)
    amp = torch.where(K2 == 0, torch.zeros_like(K2), torch.sqrt(K ** 4 * torch.exp(-2.0 * (K / 4.0) ** 2) /
                                                               torch.clamp(K2, min=1.0)))
    amp = amp * (K < 24.0)

    def noise():
        z = torch.randn(2, *shape, generator=g, device="cuda", dtype=torch.float64)
        return torch.complex(z[0], z[1]) * amp

    a = [noise() for _ in range(3)]
    dot = sum(k * v for k, v in zip(ks, a)) / torch.clamp(K2, min=1.0)
    vel = [torch.fft.ifftn(v - k * dot).real for k, v in zip(ks, a)]      # along z, y, x
    vel = [v - v.mean() for v in vel]
    urms = torch.sqrt(sum((v * v).mean() for v in vel))
    vel = [v * (0.6 / urms) for v in vel]
    s = torch.fft.ifftn(noise()).real
    rho = 1.0 + 0.05 * s / torch.sqrt((s * s).mean())
    rho = torch.clamp(rho, min=0.5)
    return _cons(rho, [vel[2], vel[1], vel[0]], rho ** gamma / gamma, gamma)


def _batch(case, seed):
    """Uneven tubes: sizes log-uniform; rarefaction, contact and shock between random states."""
    gc = torch.Generator().manual_seed(20200320)     # the sizes belong to the case, not to the inputs
    lo, hi = math.log(case["n_min"]), math.log(case["n_max"])
    n = torch.exp(lo + (hi - lo) * torch.rand(case["nprob"], generator=gc, dtype=torch.float64)).round().long()
    n = n.clamp(case["n_min"], case["n_max"])
    g = torch.Generator(device="cuda").manual_seed(1000003 * (seed + 1) + 13)
    off = torch.zeros(case["nprob"] + 1, dtype=torch.long)
    off[1:] = torch.cumsum(n, 0)
    nd, od = n.cuda(), off.cuda()
    pid = torch.repeat_interleave(torch.arange(case["nprob"], device="cuda"), nd)
    i = torch.arange(int(off[-1]), device="cuda") - od[pid]
    h = 1.0 / nd.double()
    x, hx = (i.double() + 0.5) * h[pid], h[pid]
    m = case["nprob"]
    rl, rr = (0.1 + 1.9 * _rand(g, m))[pid], (0.1 + 1.9 * _rand(g, m))[pid]
    ul, ur = (2.0 * _rand(g, m) - 1.0)[pid], (2.0 * _rand(g, m) - 1.0)[pid]
    pl, pr = (0.1 + 9.9 * _rand(g, m))[pid], (0.1 + 9.9 * _rand(g, m))[pid]
    c = (0.4 + 0.2 * _rand(g, m))[pid]
    fan, con, sho = _front(x, c - 0.2, 0.04), _front(x, c, 1.5 * hx), _front(x, c + 0.2, 0.8 * hx)
    pm, um = torch.sqrt(pl * pr), 0.5 * (ul + ur)
    rho = rl + (torch.sqrt(rl * rr) - rl) * fan + (rr * 1.2 - torch.sqrt(rl * rr)) * con - 0.2 * rr * sho
    u = ul + (um - ul) * fan + (ur - um) * sho
    p = pl + (pm - pl) * fan + (pr - pm) * sho
    return n.numpy(), pid, od, h, _cons(rho, [u], p, 1.4)


def _dt(case):
    """The fixed step of the reverse and rollout cases: CFL about 0.3 at |u| + c of about 2.5."""
    return 0.3 / (3.0 * 2.5) * (2.0 * math.pi / max(_dims(case)))


def _grid(case):
    dx, bc, gamma, grav, faces = _box(case)
    return api.EulerGrid(_dims(case), dx, bc, api.Scheme(gamma=gamma, scheme=case.get("scheme", "lad")), grav, faces)


def prepare(case, seed):
    call = case["call"]
    if call == "batch":
        n, _, _, h, U0 = _batch(case, seed)
        bs = api.BatchSolver(n, h.cpu().numpy(), [1.0] * len(n))
        return {"call": call, "solver": bs, "U0": U0, "U": torch.empty_like(U0)}
    grid = _grid(case)
    U0 = _state(case, seed)
    st = {"call": call, "grid": grid, "U0": U0}
    if call == "step":
        st["solver"] = api.Solver(grid)
        st["U"] = torch.empty_like(U0)
    elif call == "rhs":
        st["ws"] = api.alloc_workspace(grid.workspace_bytes(0), U0.device)
        st["out"] = torch.empty_like(U0)
    else:
        g = torch.Generator(device="cuda").manual_seed(77 * seed + 5)
        st["bar"] = torch.randn(U0.shape, generator=g, device="cuda", dtype=torch.float64)
        st["dt"] = _dt(case)
        if call == "adjoint":
            st["stepper"] = api.AdjointStepper(grid)
            st["out"] = torch.empty_like(U0)
        else:
            st["steps"] = case["steps"]
            st["U0"] = U0.requires_grad_(True)
    return st


def run(state):
    call = state["call"]
    if call == "step":
        U = state["U"]
        U.copy_(state["U0"])
        state["solver"].step(U)
        return {"U": U, "dt": state["solver"].dt}
    if call == "rhs":
        return api.rhs(state["grid"], state["U0"], ws=state["ws"], out=state["out"])
    if call == "batch":
        U = state["U"]
        U.copy_(state["U0"])
        state["solver"].t.zero_()
        state["solver"].step(U)
        return {"U": U, "t": state["solver"].t}
    if call == "adjoint":
        return state["stepper"].step(state["U0"], state["dt"], state["bar"], state["out"])
    out = api.rollout(state["U0"], state["grid"], state["steps"], state["dt"])
    (grad,) = torch.autograd.grad(out, state["U0"], grad_outputs=state["bar"])
    return {"U": out.detach(), "grad": grad}


def work(case):
    """Each input read once and each output written once; the arithmetic of a
    kept-stencil interface (Roe average, two six-point sums per component,
    the characteristic correction), of the cell pass and of the difference.
    The cutoff-free scheme pays the characteristic reconstruction everywhere."""
    if case["call"] == "batch":
        lo, hi = math.log(case["n_min"]), math.log(case["n_max"])
        mean = (case["n_max"] - case["n_min"]) / (hi - lo) if hi > lo else case["n_min"]
        cells, ndim = case["nprob"] * mean, 1
    else:
        n = _dims(case)
        cells, ndim = float(math.prod(n)), len(n)
    nvar = ndim + 2
    state = 8.0 * nvar * cells
    face = {1: 119, 2: 153, 3: 187}[ndim]
    if case.get("scheme") == "wenoz":
        face = {1: 174, 2: 290, 3: 341}[ndim] + 2 * nvar * 60
    rhs = cells * (ndim * face + 30 + 5 * ndim + 4 * nvar * ndim)
    call = case["call"]
    if call == "rhs":
        return {"bytes": 2 * state, "flops": rhs}
    if call in ("step", "batch"):
        return {"bytes": 2 * state, "flops": 3 * rhs}
    # a reverse sweep costs about twice its forward evaluation
    if call == "adjoint":
        return {"bytes": 3 * state, "flops": 2 * rhs + 6 * rhs}
    return {"bytes": 4 * state, "flops": case["steps"] * (6 * rhs + 6 * rhs)}


# ---------------------------------------------------------------------------
# the same results in plain binary64 torch, from the paper's equations
# ---------------------------------------------------------------------------
def _prim(U, gamma):
    rho = U[0]
    vel = [U[k] / rho for k in range(1, len(U) - 1)]
    p = (gamma - 1.0) * (U[-1] - 0.5 * rho * sum(v * v for v in vel))
    return rho, vel, p


def _weights(v, scheme):
    """omega_k (eq. 2.8-2.15, 3.1-3.4), held fixed in a derivative."""
    with torch.no_grad():
        v = [x.detach() for x in v]
        b = [13.0 / 12.0 * (v[0] - 2.0 * v[1] + v[2]) ** 2 + 0.25 * (v[0] - 4.0 * v[1] + 3.0 * v[2]) ** 2,
             13.0 / 12.0 * (v[1] - 2.0 * v[2] + v[3]) ** 2 + 0.25 * (v[1] - v[3]) ** 2,
             13.0 / 12.0 * (v[2] - 2.0 * v[3] + v[4]) ** 2 + 0.25 * (3.0 * v[2] - 4.0 * v[3] + v[4]) ** 2]
        tau = (b[2] - b[0]).abs()
        c = (0.1, 0.6, 0.3)
        chi = [tau / (x + EPS) for x in b]
        if scheme == "wenoz":
            a = [ck * (1.0 + x) for ck, x in zip(c, chi)]
        else:
            gam = [(1.0 + x) ** 6 for x in chi]
            if scheme == "lad":
                theta = 1.0 / (1.0 + torch.maximum(chi[0], torch.maximum(chi[1], chi[2])) / H_LAD)
                m = B_L + torch.floor(theta * (B_U - B_L))
            elif scheme == "teno5":
                m = torch.full_like(tau, 7.0)
            else:
                xi2, cr = 1e-6, 0.25
                ea = 0.9 * cr / (1.0 - 0.9 * cr) * xi2
                d = [v[k + 1] - v[k] for k in range(4)]
                eta = [(2.0 * (d[k] * d[k + 1]).abs() + ea) / (d[k] ** 2 + d[k + 1] ** 2 + ea) for k in range(3)]
                eta = torch.minimum(eta[0], torch.minimum(eta[1], eta[2]))
                mA = 1.0 - torch.clamp(eta / cr, max=1.0)
                m = torch.floor(10.5 - 3.5 * (1.0 - (1.0 - mA) ** 4 * (1.0 + 4.0 * mA)))
            cut = 10.0 ** -m * (gam[0] + gam[1] + gam[2])
            a = [ck * (x >= cut).double() for ck, x in zip(c, gam)]
        s = a[0] + a[1] + a[2]
        return [x / s for x in a]


def _reconstruct(v, scheme):
    w = _weights(v, scheme)
    return (w[0] * (2.0 * v[0] - 7.0 * v[1] + 11.0 * v[2]) + w[1] * (-v[1] + 5.0 * v[2] + 2.0 * v[3]) +
            w[2] * (2.0 * v[2] + 5.0 * v[3] - v[4])) / 6.0


def _face_flux(pts, d, gamma, alpha, scheme):
    """F^ from the six states of a face (lists of components), eq. 2.2-2.15 in characteristic fields."""
    nvar = len(pts[0])
    ndim = nvar - 2
    prim = [_prim(U, gamma) for U in pts]
    (ra, va, pa), (rb, vb, pb) = prim[2], prim[3]
    sa, sb = torch.sqrt(ra), torch.sqrt(rb)
    u = [(sa * x + sb * y) / (sa + sb) for x, y in zip(va, vb)]
    Hr = (sa * (pts[2][-1] + pa) / ra + sb * (pts[3][-1] + pb) / rb) / (sa + sb)
    q2 = sum(x * x for x in u)
    c2 = (gamma - 1.0) * (Hr - 0.5 * q2)
    c = torch.sqrt(c2)
    b1 = (gamma - 1.0) / c2

    def left(X):
        A = 0.5 * b1 * (0.5 * q2 * X[0] - sum(x * y for x, y in zip(u, X[1:-1])) + X[-1])
        B = 0.5 * (u[d] * X[0] - X[1 + d]) / c
        return [A + B, X[0] - 2.0 * A] + [X[1 + t] - u[t] * X[0] for t in range(ndim) if t != d] + [A - B]

    gp, gm = [], []
    for U, (rho, vel, p) in zip(pts, prim):
        F = [U[1 + d]] + [U[1 + k] * vel[d] + (p if k == d else 0.0) for k in range(ndim)] + [vel[d] * (U[-1] + p)]
        w, f = left(U), left(F)
        gp.append([0.5 * (f[s] + alpha[s] * w[s]) for s in range(nvar)])
        gm.append([0.5 * (f[s] - alpha[s] * w[s]) for s in range(nvar)])
    fc = [_reconstruct([gp[j][s] for j in range(5)], scheme) +
          _reconstruct([gm[j][s] for j in range(5, 0, -1)], scheme) for s in range(nvar)]
    mass = fc[0] + fc[1] + fc[-1]
    out = [mass]
    energy = fc[0] * (Hr - u[d] * c) + fc[-1] * (Hr + u[d] * c) + 0.5 * q2 * fc[1]
    s = 2
    for k in range(ndim):
        if k == d:
            out.append(u[k] * mass + c * (fc[-1] - fc[0]))
        else:
            out.append(u[k] * mass + fc[s])
            energy = energy + u[k] * fc[s]
            s += 1
    return out + [energy]


def _speeds(U, d, gamma):
    """The three global Lax-Friedrichs speeds of direction d, each from its first largest cell."""
    rho, vel, p = _prim(U, gamma)
    c = torch.sqrt(gamma * p / rho)
    out = []
    for lam in (vel[d] - c, vel[d], vel[d] + c):
        lam = lam.abs().reshape(-1)
        out.append(lam[int(torch.argmax(lam.detach()))])
    return out


def _direction(U, d, box, n, scheme, alpha):
    """-(F^_{i+1/2} - F^_{i-1/2}) / dx_d."""
    dx, bc, gamma, _, faces = box
    ndim, nvar, nd = len(n), len(n) + 2, n[d]
    ax = ndim - d                                   # tensor axis (0 is the component)
    i = torch.arange(-3, nd + 3, device=U.device)
    if bc[d] == PERIODIC:
        src = torch.remainder(i, nd)
    elif bc[d] == REFLECTIVE:
        src = torch.where(i < 0, -1 - i, torch.where(i >= nd, 2 * nd - 1 - i, i))
    else:
        src = i.clamp(0, nd - 1)
    P = U.index_select(ax, src)
    outside = ((i < 0) | (i >= nd)).reshape([nd + 6 if k == ax else 1 for k in range(1, ndim + 1)])
    if bc[d] == REFLECTIVE:
        sign = 1.0 - 2.0 * outside.double()
        P = torch.stack([P[v] * sign if v == 1 + d else P[v] for v in range(nvar)])
    elif bc[d] == DIRICHLET:
        low = (i < 0).reshape(outside.shape)
        two = torch.tensor(faces[d], dtype=torch.float64, device=U.device)
        face = [torch.where(low, two[0, v], two[1, v]) for v in range(nvar)]
        P = torch.stack([torch.where(outside, face[v].expand_as(P[v]), P[v]) for v in range(nvar)])
    al = [alpha[0]] + [alpha[1]] * ndim + [alpha[2]]
    pts = [list(P.narrow(ax, j, nd + 1).unbind(0)) for j in range(6)]
    F = torch.stack(_face_flux(pts, d, gamma, al, scheme))
    return (F.narrow(ax, 0, nd) - F.narrow(ax, 1, nd)) / dx[d]


def _rhs(U, box, n, scheme):
    """L(U) (eq. 2.2) and the speeds, in slabs across another direction to bound memory."""
    gamma, grav = box[2], box[3]
    ndim = len(n)
    speeds = [_speeds(U, d, gamma) for d in range(ndim)]
    R = torch.zeros_like(U)
    for d in range(ndim):
        cut = 0 if d != 0 else ndim - 1             # a direction that the sweep does not couple
        ax = ndim - cut
        if ndim == 1:
            R += _direction(U, d, box, n, scheme, speeds[d])
            continue
        cells = math.prod(n)
        per = max(1, int(n[cut] * min(1.0, 3.0e6 / cells)))
        for lo in range(0, n[cut], per):
            m = min(per, n[cut] - lo)
            part = U.narrow(ax, lo, m)
            nn = tuple(m if k == cut else v for k, v in enumerate(n))
            R.narrow(ax, lo, m).add_(_direction(part, d, box, nn, scheme, speeds[d]))
    if grav:
        for k in range(ndim):
            R[1 + k] += U[0] * grav[k]
            R[-1] += U[1 + k] * grav[k]
    return R, speeds


def _rhs_vjp(U, bar, box, n):
    """J(U)^T bar with the selections held, one direction at a time."""
    g = torch.zeros_like(U)
    for d in range(len(n)):
        X = U.detach().requires_grad_(True)
        with torch.enable_grad():
            out = _direction(X, d, box, n, "lad", _speeds(X, d, box[2]))
            (p,) = torch.autograd.grad(out, X, grad_outputs=bar)
        g += p
    return g


def _cfl(speeds, dx, cfl=0.5):
    s = [torch.maximum(a[0], a[2]) for a in speeds]
    return cfl / sum(x / h for x, h in zip(s, dx))


def _step(U, box, n, scheme, dt=None):
    L, speeds = _rhs(U, box, n, scheme)
    if dt is None:
        dt = _cfl(speeds, box[0])
    U1 = U + dt * L
    U2 = 0.75 * U + 0.25 * U1 + 0.25 * dt * _rhs(U1, box, n, scheme)[0]
    return U / 3.0 + 2.0 / 3.0 * U2 + 2.0 / 3.0 * dt * _rhs(U2, box, n, scheme)[0], dt, U1, U2


def _step_vjp(U, dt, bar, box, n):
    _, _, U1, U2 = _step(U, box, n, "lad", dt)
    b2 = 2.0 / 3.0 * bar + _rhs_vjp(U2, 2.0 / 3.0 * dt * bar, box, n)
    b1 = 0.25 * b2 + _rhs_vjp(U1, 0.25 * dt * b2, box, n)
    return bar / 3.0 + 0.75 * b2 + b1 + _rhs_vjp(U, dt * b1, box, n)


def _batch_exact(case, seed):
    n, pid, off, h, U0 = _batch(case, seed)
    nd = torch.as_tensor(n, device="cuda")
    m = len(n)
    fpid = torch.repeat_interleave(torch.arange(m, device="cuda"), nd + 1)
    foff = off[:-1] + torch.arange(m, device="cuda")
    face = torch.arange(fpid.numel(), device="cuda") - foff[fpid]
    last = (nd - 1)[fpid]
    idx = [off[:-1][fpid] + torch.minimum((face - 3 + j).clamp(min=0), last) for j in range(6)]
    left = torch.arange(pid.numel(), device="cuda") + pid

    def rhs(U):
        rho, vel, p = _prim(U, 1.4)
        c = torch.sqrt(1.4 * p / rho)
        sp = [torch.zeros(m, device="cuda", dtype=torch.float64).scatter_reduce(0, pid, x.abs(), "amax")
              for x in (vel[0] - c, vel[0], vel[0] + c)]
        F = torch.stack(_face_flux([[U[v][k] for v in range(3)] for k in idx], 0, 1.4, [a[fpid] for a in sp], "lad"))
        return (F[:, left] - F[:, left + 1]) / h[pid], sp

    L, sp = rhs(U0)
    dt = torch.minimum(0.5 * h / torch.maximum(sp[0], sp[2]), torch.ones_like(h))
    dtc = dt[pid]
    U1 = U0 + dtc * L
    U2 = 0.75 * U0 + 0.25 * U1 + 0.25 * dtc * rhs(U1)[0]
    return {"U": U0 / 3.0 + 2.0 / 3.0 * U2 + 2.0 / 3.0 * dtc * rhs(U2)[0], "t": dt}


def exact(case, seed):
    call = case["call"]
    with torch.no_grad():
        if call == "batch":
            return _batch_exact(case, seed)
        box, n, scheme = _box(case), _dims(case), case.get("scheme", "lad")
        U = _state(case, seed)
        if call == "rhs":
            return _rhs(U, box, n, scheme)[0]
        if call == "step":
            V, dt, _, _ = _step(U, box, n, scheme)
            return {"U": V, "dt": dt.reshape(1)}
        g = torch.Generator(device="cuda").manual_seed(77 * seed + 5)
        bar = torch.randn(U.shape, generator=g, device="cuda", dtype=torch.float64)
        dt = _dt(case)
        if call == "adjoint":
            return _step_vjp(U, dt, bar, box, n)
        states = [U]
        for _ in range(case["steps"]):
            states.append(_step(states[-1], box, n, scheme, dt)[0])
        for V in reversed(states[:-1]):
            bar = _step_vjp(V, dt, bar, box, n)
        return {"U": states[-1], "grad": bar}
