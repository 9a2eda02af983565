"""One geometric multigrid V-cycle and the Stokes preconditioner P_S in NumPy, written from
their definition with one small matrix per axis: no code or layout of the library.

A field is given by its rule on every axis: "per" (periodic), "cdir" / "cneu" (cell-centred
between walls, ghost value -u / +u) or "vert" (the normal velocity component, on faces 0 ..
n-1 of an axis whose faces 0 and n are walls; face 0 is stored, its row is u = f and
its value is no neighbour).  Arrays have shape n[::-1], x fastest.
"""
import numpy as np


def _second_difference(n, rule):
    M = -2.0 * np.eye(n)
    for i in range(n):
        for j in (i - 1, i + 1):
            if rule == "per":
                M[i, j % n] += 1.0
            elif 0 <= j < n:
                M[i, j] += 1.0
            elif rule != "vert":
                M[i, i] += 1.0 if rule == "cneu" else -1.0
    if rule == "vert":
        M[0, :] = 0.0
        M[:, 0] = 0.0
    return M


def _restriction(n, rule):
    R = np.zeros((n // 2, n))
    for c in range(n // 2):
        if rule != "vert":
            R[c, [2 * c, 2 * c + 1]] = 0.5
        elif c > 0:
            R[c, [2 * c - 1, 2 * c, 2 * c + 1]] = 0.25, 0.5, 0.25
    return R


def _prolongation(n, rule):
    P, nc = np.zeros((n, n // 2)), n // 2
    for i in range(n):
        c = i // 2
        if rule == "vert":
            for q in ((c,) if i % 2 == 0 else (c, c + 1)):
                if 0 < q < nc:
                    P[i, q] = 1.0 if i % 2 == 0 else 0.5
            continue
        q = c + 1 if i % 2 else c - 1
        P[i, c] += 0.75
        if rule == "per":
            P[i, q % nc] += 0.25
        elif 0 <= q < nc:
            P[i, q] += 0.25
        else:
            P[i, c] += 0.25 if rule == "cneu" else -0.25
    return P


def _along(M, a, u):
    """M applied to axis a (0: x) of u"""
    ax = u.ndim - 1 - a
    return np.moveaxis(np.tensordot(M, u, (1, ax)), 0, ax)


class Field:
    """sigma I - kappa Lap_h with the rules of one field, and its V-cycle"""

    def __init__(self, n, h, rules, sigma, kappa):
        self.n, self.rules, self.sigma, self.kh2 = tuple(n), rules, sigma, kappa / h ** 2
        d = len(n)
        self.lap = [_second_difference(m, r) for m, r in zip(n, rules)]
        idx = np.indices(self.n[::-1])[::-1]
        self.color = sum(idx) % 2
        self.face = np.zeros(self.n[::-1], bool)
        self.own = np.zeros(self.n[::-1])  # the Laplacian's diagonal
        for a in range(d):
            self.own += np.where(idx[a] == 0, -2.0 if rules[a] == "vert" else 0.0, 0.0)
            self.own += np.diag(self.lap[a])[idx[a]]
            if rules[a] == "vert":
                self.face |= idx[a] == 0
        self.singular = sigma == 0.0 and all(r in ("per", "cneu") for r in rules)
        self.coarse = None
        if all(m % 4 == 0 for m in n) and np.prod(n) > 64:
            self.coarse = Field([m // 2 for m in n], 2 * h, rules, sigma, kappa)

    def _laplacian(self, u):
        return sum(_along(M, a, u) for a, M in enumerate(self.lap))

    def residual(self, u, f):
        return np.where(self.face, f - u, f - (self.sigma * u - self.kh2 * self._laplacian(u)))

    def half_sweep(self, u, f, color):
        nb = self._laplacian(u) - sum(_along(np.diag(np.diag(M)), a, u) for a, M in enumerate(self.lap))
        new = np.where(self.face, f, (f + self.kh2 * nb) / (self.sigma - self.kh2 * self.own))
        return np.where(self.color == color, new, u)

    def vcycle(self, u, f, pre, post):
        """u: None for a start from zero"""
        zero = u is None
        if zero:
            u = np.zeros(self.n[::-1])
        if self.coarse is None:
            mean = zero and self.singular
            f = f - f.mean() if mean else f
            for _ in range(max(8, 2 * max(self.n))):
                u = self.half_sweep(self.half_sweep(u, f, 0), f, 1)
            return u - u.mean() if mean else u
        for _ in range(pre):
            u = self.half_sweep(self.half_sweep(u, f, 0), f, 1)
        r = self.residual(u, f)
        for a, (m, rule) in enumerate(zip(self.n, self.rules)):
            r = _along(_restriction(m, rule), a, r)
        e = self.coarse.vcycle(None, r, pre, post)
        for a, (m, rule) in enumerate(zip(self.n, self.rules)):
            e = _along(_prolongation(m, rule), a, e)
        u = u + e
        for _ in range(post):
            u = self.half_sweep(self.half_sweep(u, f, 1), f, 0)
        return u


def field_rules(d, walls, component):
    """component: 0 .. d-1, or None for the pressure"""
    out = []
    for a in range(d):
        if not (walls >> a) & 1:
            out.append("per")
        else:
            out.append("cneu" if component is None else "vert" if component == a else "cdir")
    return out


def stokes_pc(n, h, walls, r, eta, rho, dt, pre, post):
    """z = P_S r (d velocity components and the pressure, each of shape n[::-1])"""
    d = len(n)
    sigma = rho / dt if rho > 0 and dt > 0 else 0.0
    y = [Field(n, h, field_rules(d, walls, a), sigma, eta).vcycle(None, r[a], pre, post) for a in range(d)]
    div = 0.0
    for a in range(d):
        ax = d - 1 - a
        v = y[a].copy()
        if (walls >> a) & 1:
            np.moveaxis(v, ax, 0)[0] = 0.0  # the low wall's face; the high one wraps onto it
        div = div + np.roll(v, -1, ax) - v
    q = -div / h - r[d]
    phi = Field(n, h, field_rules(d, walls, None), 0.0, 1.0).vcycle(None, -q / h ** 2, pre, post)
    z = []
    for a in range(d):
        ax = d - 1 - a
        grad = h * (phi - np.roll(phi, 1, ax))
        if (walls >> a) & 1:
            np.moveaxis(grad, ax, 0)[0] = 0.0
        z.append(y[a] + grad)
    return z + [eta * q - (sigma * h ** 2) * phi]
