"""The right-hand side (eq. 2.2) in the host's extended precision (numpy.longdouble),
written from the paper's equations, with given selections: a reference whose own
rounding lies far below binary64's.  Boundaries: 0 periodic, 1 transmissive, 2
reflecting, 3 fixed states."""
import numpy as np

L = np.longdouble


def rhs(U, n, dx, bc, flags, gamma=1.4, faces=None):
    """dU/dt of U [nvar][..] with the selections of ``flags`` (the flag layout of teno.h)."""
    nd, nv, gm = len(n), len(n) + 2, L(gamma)
    U = U.reshape((nv,) + tuple(reversed(n))).astype(L)

    def prim(X):
        u = [X[1 + k] / X[0] for k in range(nd)]
        return u, (gm - 1) * (X[-1] - L(0.5) * X[0] * sum(v * v for v in u))

    u, p = prim(U)
    c = np.sqrt(gm * p / U[0])
    R = np.zeros_like(U)
    off = 0
    for d in range(nd):
        ax, m = nd - d, n[d]
        i = np.arange(-3, m + 3)
        al = [abs(u[d] - c).max()] + [abs(u[d]).max()] * nd + [abs(u[d] + c).max()]
        flip = np.zeros(m + 6, bool)
        if bc[d] == 0:
            src = np.mod(i, m)
        elif bc[d] == 2:
            src = i.copy()
            while ((src < 0) | (src >= m)).any():
                low = src < 0
                src, flip = np.where(low, -1 - src, src), flip ^ low
                high = src >= m
                src, flip = np.where(high, 2 * m - 1 - src, src), flip ^ high
        else:
            src = np.clip(i, 0, m - 1)
        P = np.take(U, src, axis=ax)
        shape = [m + 6 if k == ax else 1 for k in range(1, nd + 1)]
        if bc[d] == 2:
            P[1 + d] *= np.where(flip, -1, 1).astype(L).reshape(shape)
        if bc[d] == 3:
            for side, out in ((0, i < 0), (1, i >= m)):
                for v in range(nv):
                    P[v] = np.where(out.reshape(shape), L(faces[d][side][v]), P[v])
        pts = [np.stack([np.take(P[v], np.arange(j, j + m + 1), axis=nd - 1 - d) for v in range(nv)]) for j in range(6)]
        a, b = pts[2], pts[3]
        (ua, pa), (ub, pb) = prim(a), prim(b)
        sa, sb = np.sqrt(a[0]), np.sqrt(b[0])
        ut = [(sa * x + sb * y) / (sa + sb) for x, y in zip(ua, ub)]
        H = (sa * (a[-1] + pa) / a[0] + sb * (b[-1] + pb) / b[0]) / (sa + sb)
        q2 = sum(x * x for x in ut)
        c2 = (gm - 1) * (H - q2 / 2)
        cs, b1 = np.sqrt(c2), (gm - 1) / c2

        def left(X):
            A = L(0.5) * b1 * (q2 / 2 * X[0] - sum(ut[k] * X[1 + k] for k in range(nd)) + X[-1])
            B = L(0.5) * (ut[d] * X[0] - X[1 + d]) / cs
            return [A + B, X[0] - 2 * A] + [X[1 + t] - ut[t] * X[0] for t in range(nd) if t != d] + [A - B]

        W, G = [left(X) for X in pts], []
        for X in pts:
            uu, pp = prim(X)
            G.append(left([X[1 + d]] + [X[1 + k] * uu[d] + (pp if k == d else 0) for k in range(nd)] + [uu[d] * (X[-1] + pp)]))
        nif = pts[0][0].size
        sel = flags.reshape(-1)[off:off + 2 * nv * nif].reshape((nv, 2) + pts[0][0].shape)
        off += 2 * nv * nif
        f = []
        for q in range(nv):
            tot = 0
            for side, sg, order in ((0, 1, range(5)), (1, -1, range(5, 0, -1))):
                v = [L(0.5) * (G[j][q] + sg * al[q] * W[j][q]) for j in order]
                o = [((sel[q, side] >> k) & 1) * L(ck) / 10 for k, ck in enumerate((1, 6, 3))]
                tot = tot + (o[0] * (2 * v[0] - 7 * v[1] + 11 * v[2]) + o[1] * (-v[1] + 5 * v[2] + 2 * v[3]) +
                             o[2] * (2 * v[2] + 5 * v[3] - v[4])) / (6 * (o[0] + o[1] + o[2]))
            f.append(tot)
        mass = f[0] + f[1] + f[-1]
        F, en, t = [mass], f[0] * (H - ut[d] * cs) + f[-1] * (H + ut[d] * cs) + q2 / 2 * f[1], 2
        for k in range(nd):
            if k == d:
                F.append(ut[k] * mass + cs * (f[-1] - f[0]))
            else:
                F.append(ut[k] * mass + f[t])
                en = en + ut[k] * f[t]
                t += 1
        F.append(en)
        for v in range(nv):
            R[v] += (np.take(F[v], np.arange(m), axis=nd - 1 - d) - np.take(F[v], np.arange(1, m + 1), axis=nd - 1 - d)) / L(dx[d])
    return R
