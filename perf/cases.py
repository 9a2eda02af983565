"""The calls whose time this repository is judged by, measured through the public binding
``paper_1505_07865_gb300.abi``: constrained Stokes solves of every kind the library takes, the
set-up of a new geometry, time steps between walls, a mix of requests through the serving engine,
and one product with the system matrix.

Boxes are periodic with height 1 (cells h = 1 / n[1]) unless a case has walls; disks and spheres
carry surface markers at about 2h, are placed at random without overlap, and move with N(0, 1)
rigid velocities (free bodies: N(0, 1) forces and torques).  Everything is drawn from the seed.

``exact`` solves the same problem in float64 with plain torch: the periodic Stokes operators are
diagonal in the discrete Fourier basis, the marker forces follow from the Schur complement (dense
on small problems, else by conjugate gradients).
"""
import math

import numpy as np
import torch

from paper_1505_07865_gb300 import abi

DEV = "cuda"


# ---- the cases ---------------------------------------------------------------

def _eta(n1):
    """A viscosity for n1 cells per unit length, to two digits.  The momentum rows of the system scale
    with eta h^-2, and the residual that stops a solve is not weighted: with eta h^-2 of a few
    thousand, the 64^2 configuration's own value, a residual of 1e-10 is in reach on every grid."""
    return float("%.2g" % (3300.0 / n1 ** 2))


def _case(kind, n, bodies, radius, precision="mixed", mob="auto", eta=None, tol=None, kernel=4, free=0, setup=False,
          steps=0, requests=0):
    """One case.  kind: "solve", "steps", "serve" or "matvec"; n: cells; bodies of about `radius`;
    free: how many of them have a given load instead of a given velocity; setup: every pass hands the
    markers over anew, so it bins them and builds and factorises the mobility too; steps: time steps a
    pass takes; requests: solves a pass sends through the engine.  Solves go to residuals at which the
    forces, too, are right to nine digits (free bodies reach them earlier: their right-hand side holds
    the loads alone)."""
    n = list(n) + [1] * (3 - len(n))
    if tol is None:
        tol = 1e-9 if free == bodies else 3e-10 if n[2] > 1 else 1.2e-10
    return {"kind": kind, "n0": n[0], "n1": n[1], "n2": n[2], "bodies": bodies, "radius": radius, "precision": precision,
            "mob": mob, "eta": _eta(n[1]) if eta is None else eta, "tol": tol, "kernel": kernel, "free": free,
            "setup": setup, "steps": steps, "requests": requests}


def listed():
    return [
        # the smallest configuration: one disk on 64^2, all FP64, solved to 1e-10
        dict(_case("solve", (64, 64), 1, 0.1, "fp64", eta=1.0, tol=1e-10), name="disk_64_fp64"),
        # the usual 2-D solve of a batch, tabulated pair mobility; here of freely moving disks
        dict(_case("solve", (128, 128), 3, 0.1, mob="pair", free=3), name="free_disks_128"),
        # disks that move between solves: the set-up belongs to every pass
        dict(_case("solve", (256, 256), 5, 0.1, mob="pair", setup=True), name="moving_disks_256"),
        # the largest 2-D problem of the batch, crowded
        dict(_case("solve", (512, 512), 8, 0.1, mob="pair"), name="disks_512"),
        # flow past a disk in a channel with no-slip walls: explicit advection, one solve per time step
        dict(_case("steps", (128, 64), 1, 0.12, eta=0.4, tol=5e-12, steps=4), name="channel_steps_128x64"),
        # a batch of 2-D requests of different sizes through the serving engine
        dict(_case("serve", (128, 128), 4, 0.08, mob="pair", requests=12), name="serve_2d_mix"),
        # the smallest grid of the 3-D stream, with the six-point kernel
        dict(_case("solve", (64, 64, 64), 1, 0.15, kernel=6), name="sphere_64_bkp6"),
        # all-FP64 solve on a box with unequal sides
        dict(_case("solve", (96, 64, 48), 2, 0.15, "fp64"), name="box_96x64x48_fp64"),
        # a 3-D request of the stream: several bodies, new geometry, its mobility built and factorised
        dict(_case("solve", (96, 96, 96), 4, 0.1, mob="pair", setup=True), name="request_96"),
        # the benchmark's problem: one sphere on 128^3, markers handed over for every solve
        dict(_case("solve", (128, 128, 128), 1, 0.1, setup=True), name="sphere_128"),
        # the largest grid of the 3-D stream
        dict(_case("solve", (192, 192, 192), 3, 0.08), name="spheres_192"),
        # one product with the system matrix (FP64), as a caller's own iteration needs it
        dict(_case("matvec", (128, 128, 128), 4, 0.1, "fp64"), name="matvec_128"),
    ]


def draw(rng):
    """A case of the ranges above; cells per axis are m 2^p with a small odd m, as the multigrid needs them."""
    kind = rng.choice(["solve2", "solve2", "solve2", "solve3", "solve3", "solve3", "fp64", "steps", "serve", "matvec"])

    def size(lo, hi, odd):
        fits = sorted({m << p for m in odd for p in range(1, 10) if lo <= m << p <= hi})
        x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        return min(fits, key=lambda f: abs(math.log(f / x)))

    radius = round(rng.uniform(0.07, 0.13), 3)
    if kind == "solve2":
        n1 = size(48, 512, (1, 3, 5, 7, 9, 11))
        n0 = n1 * rng.choice([1, 1, 2]) if n1 <= 256 else n1
        nb = rng.randint(2, 8) if n1 >= 128 else rng.randint(1, 3)
        return _case("solve", (n0, n1), nb, min(radius, 0.1) if nb > 5 else radius, mob="pair",
                     free=rng.choice([0, 0, nb]) if n1 <= 160 else 0, setup=rng.random() < 0.5)
    if kind == "solve3":
        n1 = size(32, 160, (1, 3, 5))
        n0 = n1 * rng.choice([1, 1, 2]) if n1 <= 64 else n1
        nb = rng.randint(1, 4) if n1 <= 96 else 1
        return _case("solve", (n0, n1, n1), nb, radius, mob=rng.choice(["auto", "auto", "pair"]),
                     kernel=rng.choice([4, 4, 6]), free=rng.choice([0, 0, nb]) if nb < 3 else 0, setup=rng.random() < 0.5)
    if kind == "fp64":
        if rng.random() < 0.5:
            n1 = size(32, 128, (1, 3, 5, 7))
            return _case("solve", (n1, n1), rng.randint(1, 3) if n1 >= 64 else 1, radius, "fp64", mob="pair")
        n1 = size(32, 64, (1, 3, 5))
        return _case("solve", (n1 * rng.choice([1, 2]), n1, n1), rng.randint(1, 2), radius, "fp64")
    if kind == "steps":
        n1 = size(40, 128, (1, 3, 5))
        return _case("steps", (2 * n1, n1), 1, radius, eta=rng.choice([0.4, 1.0]), tol=5e-12, steps=rng.randint(2, 4))
    if kind == "serve":
        return _case("serve", (size(64, 160, (1, 3, 5)),) * 2, rng.randint(2, 5), min(radius, 0.1), mob="pair",
                     requests=rng.randint(4, 16))
    n1 = size(32, 160, (1, 3, 5))
    return _case("matvec", (n1, n1, n1) if rng.random() < 0.7 else (4 * n1, 2 * n1), rng.randint(1, 4), radius, "fp64")


# ---- geometry ------------------------------------------------------------------

def _dim(case):
    return 2 if case["n2"] == 1 else 3


def _cells(case):
    return tuple(case[k] for k in ("n0", "n1", "n2")[:_dim(case)])


def _ring(radius, h):
    m = max(3, round(math.pi * radius / h))
    t = 2.0 * np.pi * np.arange(m) / m
    return radius * np.stack([np.cos(t), np.sin(t)], axis=1)


def _shell(radius, h):
    """Golden-spiral points on a sphere, one per 2h-triangle lattice cell of its area."""
    m = max(12, round(4.0 * math.pi * radius ** 2 / (math.sqrt(3.0) / 2.0 * (2.0 * h) ** 2)))
    i = np.arange(m)
    z = 1.0 - (2.0 * i + 1.0) / m
    s, p = np.sqrt(1.0 - z * z), np.pi * (3.0 - math.sqrt(5.0)) * i
    return radius * np.stack([s * np.cos(p), s * np.sin(p), z], axis=1)


def _place(rng, radii, L, h, walled):
    """Random centres with at least 4h between the bodies (the kernel's support); a placement in which
    a body finds no room is begun anew."""
    if walled:
        return [L * np.array([rng.uniform(0.35, 0.5), rng.uniform(0.4, 0.6)])]
    while True:
        cs = []
        for r in radii:
            for _ in range(500):
                c = rng.uniform(0.0, 1.0, len(L)) * L
                if all(np.linalg.norm((c - q + 0.5 * L) % L - 0.5 * L) >= r + s + 4.0 * h for q, s in zip(cs, radii)):
                    cs.append(c)
                    break
            else:
                break
        if len(cs) == len(radii):
            return cs


class _Problem:
    """Box, bodies and loads of a case for one seed."""

    def __init__(self, case, seed, n=None, bodies=None):
        rng = np.random.default_rng([1505, int(seed)])
        self.n = tuple(n or _cells(case))
        self.d = len(self.n)
        self.h = 1.0 / self.n[1]
        self.L = tuple(m * self.h for m in self.n)
        self.eta, self.kernel = case["eta"], case["kernel"]
        self.walled = case["kind"] == "steps"
        self.rho, self.dt = (1.0, 0.25 * self.h) if self.walled else (0.0, 0.0)
        nr = 3 if self.d == 2 else 6
        B = bodies or case["bodies"]
        radii = [case["radius"] * (1.0 - 0.04 * (b % 4)) for b in range(B)]
        self.rels = [_ring(r, self.h) if self.d == 2 else _shell(r, self.h) for r in radii]
        self.centers = _place(rng, radii, np.array(self.L), self.h, self.walled)
        self.free = [b < case["free"] for b in range(B)]
        self.UO = rng.standard_normal((B, nr))
        if self.walled:
            self.UO[:] = 0.0
        self.body = np.repeat(np.arange(B), [len(r) for r in self.rels])
        self.rel = np.concatenate(self.rels)
        self.q = np.concatenate([c + r for c, r in zip(self.centers, self.rels)])
        self.N, self.ncell = len(self.q), int(np.prod(self.n))


class _Grid:
    """A grid handle with its bodies; destroyed with the object."""

    def __init__(self, case, P):
        self.P, self.case, self.h = P, case, None
        bc, per = [], not P.walled
        for a in range(P.d):
            bc += [abi.PERIODIC] * 2 if per else ([abi.VELOCITY] * 2 if a == 0 else [abi.NOSLIP] * 2)
        self.h = abi.create_grid(P.d, P.n, P.L, bc=bc, eta=P.eta, rho=P.rho, dt=P.dt,
                                 kernel=abi.KERNEL_BKP6 if P.kernel == 6 else abi.KERNEL_PESKIN4,
                                 precision=abi.FP64 if case["precision"] == "fp64" else abi.MIXED)
        if P.walled:
            y = (np.arange(P.n[1]) + 0.5) * P.h
            prof = np.zeros((2, P.n[1]))
            prof[0] = 4.0 * y * (1.0 - y)
            abi.set_boundary_velocity(self.h, 0, prof)
            abi.set_boundary_velocity(self.h, 1, prof)
        for c, f in zip(P.centers, P.free):
            abi.add_body(self.h, c, kinematics=abi.FREE if f else abi.PRESCRIBED)
        self.opts = _opts(case)
        self.markers()
        abi.prepare(self.h, self.opts)
        self.v = torch.empty(P.d * P.ncell, dtype=torch.float64, device=DEV)
        self.p = torch.empty(P.ncell, dtype=torch.float64, device=DEV)

    def markers(self):
        for b, r in enumerate(self.P.rels):
            abi.set_markers(self.h, b, r)

    def results(self):
        abi.get_fields(self.h, self.v, self.p)
        lam, ft = abi.get_forces(self.h, self.P.d)
        out = {"v": self.v, "p": self.p, "lam": lam, "ft": ft}
        if any(self.P.free):
            out["U"] = abi.get_body_velocities(self.h, self.P.UO)
        return out

    def __del__(self):
        if self.h is not None:
            abi.destroy_grid(self.h)
            self.h = None


def _opts(case):
    o = abi.solve_opts_default()
    o.tol = case["tol"]
    o.mob_model = abi.MOB_PAIR if case["mob"] == "pair" else abi.MOB_AUTO
    return o


def _requests(case, seed):
    """The engine's mix: half, once and twice the case's cells per axis, two to `bodies` disks each."""
    rng = np.random.default_rng(41)  # the sizes are the case's, the placements and velocities the seed's
    out = []
    for i in range(case["requests"]):
        m = (case["n0"] // 2, case["n0"], 2 * case["n0"])[i % 3]
        out.append(_Problem(dict(case, eta=_eta(m)), 1000 * int(seed) + i, (m, m), int(rng.integers(2, case["bodies"] + 1))))
    return out


class _Serving:
    def __init__(self, case, seed):
        self.reqs, self.opts = _requests(case, seed), _opts(case)
        self.server = abi.Server(slots=8, budget_bytes=64 << 30)

    def __del__(self):
        self.server.close()


def prepare(case, seed):
    if case["kind"] == "serve":
        return _Serving(case, seed)
    G = _Grid(case, _Problem(case, seed))
    if case["kind"] == "steps":
        # the state that the march starts from: the inflow profile everywhere, slightly disturbed
        gen = torch.Generator(device=DEV).manual_seed(int(seed))
        n0, n1 = G.P.n
        y = (torch.arange(n1, device=DEV, dtype=torch.float64) + 0.5) / n1
        G.v0 = torch.zeros(2, n1, n0, dtype=torch.float64, device=DEV)
        G.v0[0] = (4.0 * y * (1.0 - y))[:, None]
        G.v0 += 0.02 * torch.randn(G.v0.shape, generator=gen, dtype=torch.float64, device=DEV)
        G.v0 = G.v0.reshape(-1).contiguous()
    if case["kind"] == "matvec":
        gen = torch.Generator(device=DEV).manual_seed(int(seed))
        G.x = torch.randn(abi.sizes(G.h)[0], generator=gen, dtype=torch.float64, device=DEV)
        G.y = torch.empty_like(G.x)
    torch.cuda.synchronize()
    return G


def run(state):
    if isinstance(state, _Serving):
        tickets = [state.server.submit(P.n, P.L, P.centers, P.rels, P.UO, eta=P.eta, opts=state.opts) for P in state.reqs]
        done = [state.server.poll(t) for t in tickets]
        return [{"lam": r["lam"], "ft": r["ft"]} for r in done]
    G, kind = state, state.case["kind"]
    if kind == "matvec":
        abi.apply_system(G.h, G.x, G.y)
        return G.y
    if kind == "steps":
        abi.set_velocity(G.h, G.v0)
        abi.advance(G.h, G.P.UO, G.case["steps"], opts=G.opts)
        return G.results()
    if G.case["setup"]:
        G.markers()
    abi.solve_coupled(G.h, G.P.UO, opts=G.opts)
    return G.results()


def work(case):
    """What a solve cannot do without: each of its inputs and results once, and per outer iteration at
    least one product with the matrix and one use of the preconditioner, a read and a write of a vector
    each in the precision they run in (20 iterations of a solve, 10 of a time step started from the last)."""
    d, cells = _dim(case), float(np.prod(_cells(case)))
    vec = (d + 1) * cells
    pc = 8.0 if case["precision"] == "fp64" else 4.0
    if case["kind"] == "matvec":
        return {"bytes": 16.0 * vec, "flops": (13.0 * d + 2 * d) * cells}
    per = vec * (16.0 + 2.0 * pc)
    flops = (13.0 * d + 2 * d) * cells * 3.0
    if case["kind"] == "serve":  # half, once and twice the cells per axis in turn
        k = case["requests"] * (0.25 + 1.0 + 4.0) / 3.0
        return {"bytes": 20.0 * per * k, "flops": 20.0 * flops * k}
    its = 10.0 * case["steps"] if case["kind"] == "steps" else 20.0
    return {"bytes": its * per + 8.0 * vec, "flops": its * flops}


# ---- the same in float64 by Fourier transforms -----------------------------------

def _phi4(r):
    """4-point kernel weights at nodes floor - 1 .. floor + 2 for the fractions r in [0, 1)."""
    def inner(x):
        return (3.0 - 2.0 * x + torch.sqrt(1.0 + 4.0 * x - 4.0 * x * x)) / 8.0

    def outer(x):
        return (5.0 - 2.0 * x - torch.sqrt((-7.0 + 12.0 * x - 4.0 * x * x).clamp(min=0.0))) / 8.0

    return torch.stack([outer(1.0 + r), inner(r), inner(1.0 - r), outer(2.0 - r)], dim=-1)


def _phi6(r):
    """Weights of the six-point kernel at nodes floor - 2 .. floor + 3: the family that the moment and
    even-odd conditions leave, p + t z with z = (1, -3, 2, 2, -3, 1), fixed by the sum of squares; the
    root that vanishes at r = 0."""
    K = 59.0 / 60.0 - math.sqrt(29.0) / 20.0
    x = r[..., None] - torch.arange(-2, 4, dtype=r.dtype, device=r.device)
    one = torch.ones_like(x)
    sgn = torch.tensor([1.0, -1.0, 1.0, -1.0, 1.0, -1.0], dtype=r.dtype, device=r.device).expand_as(x)
    last = torch.zeros_like(x)
    last[..., 5] = 1.0  # the member of the family with weight 0 at the last node
    A = torch.stack([one, sgn, x, x ** 2, x ** 3, last], dim=-2)
    b = torch.zeros_like(x)
    b[..., 0], b[..., 3] = 1.0, K
    p = torch.linalg.solve(A, b)
    z = torch.tensor([-1.0, 3.0, -2.0, -2.0, 3.0, -1.0], dtype=r.dtype, device=r.device).neg()
    p0 = (0.625 - 0.25 * K, 0.25, 0.125 * K - 0.0625)  # weights at distance 0, 1, 2 for r = 0
    C = p0[0] ** 2 + 2.0 * p0[1] ** 2 + 2.0 * p0[2] ** 2
    a, hb, c = float((z * z).sum()), (p * z).sum(-1), (p * p).sum(-1) - C
    s = torch.sqrt((hb * hb - a * c).clamp(min=0.0))
    t = torch.where(hb >= 0, -c / (hb + s).clamp(min=1e-300), (s - hb) / a)
    return p + t[..., None] * z


class _Exact:
    def __init__(self, P):
        self.P, d = P, P.d
        f8 = dict(dtype=torch.float64, device=DEV)
        self.shape = P.n[::-1]
        th = []
        for a in range(d):
            s = [1] * d
            s[d - 1 - a] = P.n[a]
            th.append((2.0 * math.pi * torch.arange(P.n[a], **f8) / P.n[a]).reshape(s))
        self.G = [(1.0 - torch.exp(-1j * t)) / P.h for t in th]
        self.D = [(torch.exp(1j * t) - 1.0) / P.h for t in th]
        s2 = sum((4.0 * torch.sin(t / 2.0) ** 2).expand(self.shape) for t in th) / P.h ** 2
        self.zero = (0,) * d
        self.s2 = s2.clone()
        self.s2[self.zero] = 1.0
        self.rel = torch.tensor(P.rel, **f8)
        self.body = torch.tensor(P.body, device=DEV)
        q = torch.tensor(P.q, **f8)
        W = 6 if P.kernel == 6 else 4
        self.cell, self.w = [], []  # per component: [N, W^d] cells and weights
        for a in range(d):
            cell = torch.zeros(P.N, 1, dtype=torch.int64, device=DEV)
            wt = torch.ones(P.N, 1, **f8)
            stride = 1
            for b in range(d):
                s = q[:, b] / P.h - (0.0 if a == b else 0.5)
                fl = torch.floor(s)
                w1 = (_phi6 if W == 6 else _phi4)(s - fl)
                j = torch.remainder(fl.to(torch.int64)[:, None] - (W // 2 - 1) + torch.arange(W, device=DEV), P.n[b])
                cell = (cell[:, None, :] + (j * stride)[:, :, None]).reshape(P.N, -1)
                wt = (wt[:, None, :] * w1[:, :, None]).reshape(P.N, -1)
                stride *= P.n[b]
            self.cell.append(cell)
            self.w.append(wt)

    def J(self, v):
        return torch.stack([(self.w[a] * v[a].reshape(-1)[self.cell[a]]).sum(-1) for a in range(self.P.d)], dim=-1)

    def S(self, lam):
        """S~ lam: the force density without its mean."""
        out, vol = [], float(np.prod(self.P.L))
        for a in range(self.P.d):
            f = torch.zeros(self.P.ncell, dtype=torch.float64, device=DEV)
            f.index_add_(0, self.cell[a].reshape(-1), (self.w[a] * lam[:, a, None]).reshape(-1))
            out.append((f / self.P.h ** self.P.d - lam[:, a].sum() / vol).reshape(self.shape))
        return out

    def fluid(self, f):
        """(v, p) of the unconstrained problem."""
        fh = [torch.fft.fftn(x) for x in f]
        ph = -sum(self.D[a] * fh[a] for a in range(self.P.d)) / self.s2
        ph[self.zero] = 0.0
        v = []
        for a in range(self.P.d):
            vh = (fh[a] - self.G[a] * ph) / (self.P.eta * self.s2)
            vh[self.zero] = 0.0
            v.append(torch.fft.ifftn(vh).real)
        return v, torch.fft.ifftn(ph).real

    def M(self, lam):
        return self.J(self.fluid(self.S(lam))[0])

    def inv(self, rhs):
        """M^-1 of the columns of rhs [N, d, k]: dense while that is small, else conjugate gradients."""
        N, d, k = rhs.shape
        if N * d <= 700:
            cols = torch.eye(N * d, dtype=torch.float64, device=DEV).reshape(N * d, N, d)
            A = torch.stack([self.M(c).reshape(-1) for c in cols], dim=1)
            return torch.linalg.solve(0.5 * (A + A.T), rhs.reshape(N * d, k)).reshape(N, d, k)
        out = []
        for c in range(k):
            b = rhs[:, :, c]
            x, r = torch.zeros_like(b), b.clone()
            p, rr = r.clone(), float((r * r).sum())
            stop = 1e-26 * rr
            for _ in range(2000):
                if rr <= stop:
                    break
                Ap = self.M(p)
                al = rr / float((p * Ap).sum())
                x += al * p
                r -= al * Ap
                new = float((r * r).sum())
                p = r + (new / rr) * p
                rr = new
            out.append(x)
        return torch.stack(out, dim=-1)

    def K(self, U):
        """Marker velocities of the rigid velocities U [B, nr]."""
        u, r = U[self.body], self.rel
        if self.P.d == 2:
            return torch.stack([u[:, 0] - u[:, 2] * r[:, 1], u[:, 1] + u[:, 2] * r[:, 0]], dim=-1)
        return u[:, :3] + torch.linalg.cross(u[:, 3:], r)

    def KT(self, lam):
        r, B = self.rel, len(self.P.centers)
        if self.P.d == 2:
            row = torch.cat([lam, (r[:, 0] * lam[:, 1] - r[:, 1] * lam[:, 0])[:, None]], dim=1)
        else:
            row = torch.cat([lam, torch.linalg.cross(r, lam)], dim=1)
        return torch.zeros(B, row.shape[1], dtype=torch.float64, device=DEV).index_add_(0, self.body, row)

    def solve(self):
        P = self.P
        UO = torch.tensor(P.UO, dtype=torch.float64, device=DEV)
        free = torch.tensor(P.free, device=DEV)
        U = torch.where(free[:, None], torch.zeros_like(UO), UO)
        rhs = self.K(U)[:, :, None]
        nr, fb = UO.shape[1], torch.nonzero(free).reshape(-1).tolist()
        for b in fb:
            for c in range(nr):
                e = torch.zeros_like(UO)
                e[b, c] = 1.0
                rhs = torch.cat([rhs, self.K(e)[:, :, None]], dim=2)
        X = self.inv(rhs)
        lam = X[:, :, 0]
        if fb:
            R = torch.stack([self.KT(X[:, :, 1 + c])[fb].reshape(-1) for c in range(len(fb) * nr)], dim=1)
            u = torch.linalg.solve(R, UO[fb].reshape(-1) - self.KT(lam)[fb].reshape(-1))
            lam = lam + (X[:, :, 1:] * u).sum(-1)
            U = U.clone()
            U[fb] = u.reshape(len(fb), nr)
        v, p = self.fluid(self.S(lam))
        out = {"v": torch.cat([x.reshape(-1) for x in v]), "p": p.reshape(-1), "lam": lam, "ft": self.KT(lam)}
        if fb:
            out["U"] = U
        return out

    def matvec(self, x):
        P, n = self.P, self.P.ncell
        v = [x[a * n:(a + 1) * n].reshape(self.shape) for a in range(P.d)]
        p = x[P.d * n:(P.d + 1) * n].reshape(self.shape)
        f = self.S(x[(P.d + 1) * n:].reshape(P.N, P.d))
        out, div = [], torch.zeros_like(p)
        for a in range(P.d):
            lap = -2.0 * P.d * v[a]
            for b in range(P.d):
                lap = lap + torch.roll(v[a], 1, P.d - 1 - b) + torch.roll(v[a], -1, P.d - 1 - b)
            out.append((-P.eta / P.h ** 2 * lap + (p - torch.roll(p, 1, P.d - 1 - a)) / P.h - f[a]).reshape(-1))
            div += (torch.roll(v[a], -1, P.d - 1 - a) - v[a]) / P.h
        return torch.cat(out + [-div.reshape(-1), -self.J(v).reshape(-1)])


def exact(case, seed):
    """None for the time steps: walls have no Fourier form."""
    if case["kind"] == "steps":
        return None
    if case["kind"] == "serve":
        done = [_Exact(P).solve() for P in _requests(case, seed)]
        return [{"lam": r["lam"], "ft": r["ft"]} for r in done]
    E = _Exact(_Problem(case, seed))
    if case["kind"] == "matvec":
        gen = torch.Generator(device=DEV).manual_seed(int(seed))
        size = (E.P.d + 1) * E.P.ncell + E.P.N * E.P.d
        return E.matvec(torch.randn(size, generator=gen, dtype=torch.float64, device=DEV))
    return E.solve()
