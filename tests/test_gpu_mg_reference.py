"""The V-cycle, P_S and the inner solve against restatements of their own: NumPy per-axis
matrices (_mg_reference) for the first two, least squares over the P_S directions in
FP64 for the last.  Every path of the V-cycle is reached: the one-block tail alone,
one-launch legs, half sweeps per launch, the 3-D split layout and cluster kernel,
stacked velocity components with walls on one, several or all axes.

Tolerances.  A half sweep's update has 2D + 2 operations and does not amplify earlier
errors (the operators are diagonally dominant); a cycle updates a cell at most about 100
times, coarsest level included: 800 units of rounding of the largest value, 9e-14 in FP64
and 5e-5 in FP32, asserted as 1e-12 and 1e-4.  P_S divides a difference of velocities by h
once: the same twice over.  Inner solve: the minimiser over at most four directions whose
images have a condition below 1e3, through its normal equations: 1e6 eps = 2e-10 in FP64
(1e-9 asserted); in FP32 the products are rounded, 6e-8 times that condition (1e-4 asserted).
"""
import numpy as np
import pytest

from ._mg_reference import Field, field_rules, stokes_pc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [(4, 4), (8, 8), (16, 8), (4, 64), (24, 40), (44, 44), (72, 40), (144, 80), (8, 8, 8), (24, 16, 32), (40, 40, 40),
         (16, 64, 8)]


@pytest.fixture(scope="module")
def abi():
    from paper_1505_07865_gb300 import abi as a

    assert torch.cuda.is_available()
    return a


def _grid(abi, n, walls, precision, eta=1.0, rho=0.0, dt=0.0):
    bc = []
    for a in range(len(n)):
        bc += [abi.NOSLIP if (walls >> a) & 1 else abi.PERIODIC] * 2
    return abi.create_grid(len(n), n, [m / n[0] for m in n], bc=bc, eta=eta, rho=rho, dt=dt,
                           precision=getattr(abi, precision))


def _dev(a):
    return torch.tensor(np.ascontiguousarray(a).ravel(), device="cuda")


@pytest.mark.parametrize("sigma", [0.0, 250.0])
@pytest.mark.parametrize("walls", [0, 1, 2, 7])
@pytest.mark.parametrize("n", SIZES, ids=lambda n: "x".join(map(str, n)))
def test_vcycle_of_a_pressure_like_field(abi, n, walls, sigma):
    walls &= (1 << len(n)) - 1
    rng = np.random.default_rng(2)
    f, u = rng.standard_normal(n[::-1]), rng.standard_normal(n[::-1])
    if sigma == 0.0:
        f -= f.mean()
    ref = Field(n, 1.0 / n[0], field_rules(len(n), walls, None), sigma, 1.3).vcycle(u, f, 2, 2).ravel()
    for precision, tol in (("FP64", 1e-12), ("MIXED", 1e-4)):
        G = _grid(abi, n, walls, precision)
        try:
            out = _dev(u)
            abi.op_vcycle(G, sigma, 1.3, _dev(f), out, 1)
            err = np.abs(out.cpu().numpy() - ref).max() / np.abs(ref).max()
        finally:
            abi.destroy_grid(G)
        assert err <= tol, (precision, err)


@pytest.mark.parametrize("steady", [True, False])
@pytest.mark.parametrize("walls", [0, 1, 2, 7])
@pytest.mark.parametrize("n", SIZES, ids=lambda n: "x".join(map(str, n)))
def test_stokes_preconditioner(abi, n, walls, steady):
    _check_pc(abi, n, walls & ((1 << len(n)) - 1), steady, 2, 2)


@pytest.mark.parametrize("walls", [0, 7])
@pytest.mark.parametrize("pre,post", [(1, 1), (3, 2), (1, 3), (0, 2), (4, 1), (2, 0)])
@pytest.mark.parametrize("n", [(72, 40), (24, 16, 32)], ids=["2d", "3d"])
def test_other_sweep_counts(abi, n, pre, post, walls):
    _check_pc(abi, n, walls & ((1 << len(n)) - 1), True, pre, post)


def _check_pc(abi, n, walls, steady, pre, post):
    d = len(n)
    eta, rho, dt = 0.8, (0.0 if steady else 1.0), (0.0 if steady else 0.002)
    r = np.random.default_rng(7).standard_normal((d + 1,) + n[::-1])
    ref = stokes_pc(n, 1.0 / n[0], walls, r, eta, rho, dt, pre, post)
    for precision, tol in (("FP64", 2e-12), ("MIXED", 2e-4)):
        G = _grid(abi, n, walls, precision, eta, rho, dt)
        try:
            if (pre, post) != (2, 2):  # a solve sets the sweep counts
                _one_step(abi, G, n, np.zeros((d,) + n[::-1]), 1, pre, post)
            z = torch.zeros(r.size, dtype=torch.float64, device="cuda")
            abi.op_stokes_pc(G, _dev(r), z)
            got = z.cpu().numpy().reshape(r.shape)
        finally:
            abi.destroy_grid(G)
        for c in range(d + 1):
            err = np.abs(got[c] - ref[c]).max() / np.abs(ref[c]).max()
            assert err <= tol, (precision, c, err)


def _one_step(abi, G, n, force, n_s, pre=2, post=2):
    """one outer step for a body at rest (or moving, without a force) in the middle"""
    d = len(n)
    h = 1.0 / n[0]
    bid = abi.add_body(G, [0.5 * m * h for m in n])
    abi.set_markers(G, bid, np.array([[1.5 * h] + [0.0] * (d - 1), [-1.5 * h] + [0.0] * (d - 1)]))
    o = abi.solve_opts_default()
    o.tol, o.max_iters, o.n_s, o.mg_pre, o.mg_post = 1e-14, 1, n_s, pre, post
    uo = np.zeros(3 if d == 2 else 6)
    uo[0] = 0.0 if np.any(force) else 1.0
    assert abi.solve_coupled(G, uo, g=force.ravel(), opts=o).iters == 1


@pytest.mark.parametrize("precision,tol", [("FP64", 1e-9), ("MIXED", 1e-4)])
@pytest.mark.parametrize("n_s", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("n,walls", [((24, 40), 0), ((72, 40), 3), ((24, 16, 32), 0), ((16, 16, 16), 4), ((40, 40, 40), 0)])
def test_inner_solve_minimises_the_residual(abi, n, walls, n_s, precision, tol):
    """One outer step without a body's motion leaves a multiple of the inner solve's result: the
    combination of n_s P_S directions whose fluid residual is smallest (five: the general Arnoldi form)."""
    d, nc = len(n), int(np.prod(n))
    force = np.random.default_rng(3).standard_normal((d,) + n[::-1])
    for a in range(d):
        if (walls >> a) & 1:
            np.moveaxis(force[a], d - 1 - a, 0)[0] = 0.0
        if walls == 0:
            force[a] -= force[a].mean()
    G = _grid(abi, n, walls, precision, eta=1.0 / n[0] ** 2)
    try:
        _one_step(abi, G, n, force, n_s)
        v, p = np.zeros(d * nc), np.zeros(nc)
        abi.get_fields(G, v, p)
        nS = (d + 1) * nc
        b = torch.zeros(nS, dtype=torch.float64, device="cuda")
        b[:d * nc] = _dev(force)
        Z, W, r = [], [], b / b.norm()
        for _ in range(n_s):
            z = torch.zeros(nS, dtype=torch.float64, device="cuda")
            abi.op_stokes_pc(G, r, z)
            x = torch.zeros(abi.sizes(G)[0], dtype=torch.float64, device="cuda")
            y = torch.empty_like(x)
            x[:nS] = z
            abi.apply_system(G, x, y)
            Z.append(z)
            W.append(y[:nS].clone())
            Q = torch.linalg.qr(torch.stack([b] + W, 1))[0]  # the next direction starts at the new part of L z
            r = Q[:, -1].contiguous()
        c = torch.linalg.lstsq(torch.stack(W, 1).cpu(), b.cpu()[:, None], driver="gelsd").solution[:, 0]
        ref = (torch.stack(Z, 1).cpu() @ c).numpy().reshape(d + 1, nc)
    finally:
        abi.destroy_grid(G)
    got = np.concatenate([v, p]).reshape(d + 1, nc)
    for a in range(d + 1):
        if a == d or walls == 0:
            ref[a] -= ref[a].mean()
    got, ref = got.ravel(), ref.ravel()
    got = got * (got @ ref) / (got @ got)
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)
