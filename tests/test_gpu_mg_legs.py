"""The fused multigrid kernels against the per-level ones: a 2-D level's legs in
one launch each and the one-block tail, at sizes where tiles, halos and pairs of
cells do not fit evenly, for both precisions.

Reference: ibr_op_vcycle_noalloc (FP64), which has no temporaries for the legs: it runs
the per-level kernels down to the one-block tail, and the tail itself on levels of at
most 4096 cells (test_gpu_mg_reference.py pins that one independently).  The kernels apply the same
formulas in the same order up to the association of two sums, so FP64 agrees to
1e-13 of the largest value after two cycles of a contraction; FP32 rounding of
about 30 operations per cell and level gives 1e-5.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def abi():
    from paper_1505_07865_gb300 import abi as a

    assert torch.cuda.is_available()
    return a


def _problem(n, sigma, seed):
    rng = np.random.default_rng(seed)
    f = rng.standard_normal(int(np.prod(n)))
    if sigma == 0.0:
        f -= f.mean()
    u = rng.standard_normal(f.size)
    return torch.tensor(f, device="cuda"), torch.tensor(u - u.mean(), device="cuda")


def _vcycles(abi, n, precision, sigma, f, u, bc=None, k=2):
    G = abi.create_grid(len(n), n, [m / n[0] for m in n], bc=bc, precision=precision)
    try:
        out = u.clone()
        abi.op_vcycle(G, sigma, 1.3, f, out, k)
        torch.cuda.synchronize()
    finally:
        abi.destroy_grid(G)
    return out


@pytest.mark.parametrize("sigma", [0.0, 250.0])
@pytest.mark.parametrize("n", [(8, 8), (16, 8), (24, 40), (44, 44), (72, 40), (144, 80), (96, 256), (8, 8, 8),
                               (24, 16, 32), (40, 40, 40), (16, 16, 16)])
def test_periodic_matches_per_level_kernels(abi, n, sigma):
    f, u = _problem(n, sigma, 5)
    ref = u.clone()
    abi.op_vcycle_noalloc(len(n), n, [m / n[0] for m in n], sigma, 1.3, f, ref, 2)
    top = float(ref.abs().max())
    assert float((_vcycles(abi, n, abi.FP64, sigma, f, u) - ref).abs().max()) <= 1e-13 * top
    assert float((_vcycles(abi, n, abi.MIXED, sigma, f, u) - ref).abs().max()) <= 1e-5 * top


def _neumann_residual(f, u, n, walls, h, sigma, kappa):
    """f - (sigma u - kappa Lap u), wrapped on periodic axes and mirrored at walls"""
    u = u.reshape(n[::-1])
    lap = np.zeros_like(u)
    for a in range(len(n)):
        pad = [(0, 0)] * len(n)
        pad[len(n) - 1 - a] = (1, 1)
        e = np.pad(u, pad, mode="edge" if (walls >> a) & 1 else "wrap")
        lap += np.diff(e, n=2, axis=len(n) - 1 - a)
    return f.reshape(n[::-1]) - (sigma * u - kappa / h ** 2 * lap)


@pytest.mark.parametrize("precision", ["FP64", "MIXED"])
@pytest.mark.parametrize("n", [(16, 8), (44, 44), (24, 40), (72, 40), (144, 80), (24, 16, 32)])
@pytest.mark.parametrize("walls", [1, 2, 3])
def test_wall_cycles_contract(abi, n, walls, precision):
    """with walls there is no second path to compare with: a V-cycle that reads a
    wrong neighbour contracts towards something else, so the residual of the
    stencil (formed here) has to fall by a factor of four per cycle"""
    bc = []
    for a in range(len(n)):
        bc += [abi.NOSLIP if (walls >> a) & 1 else abi.PERIODIC] * 2
    f, u = _problem(n, 300.0, 6)
    res = []
    for k in range(4):
        out = u.cpu().numpy() if k == 0 else _vcycles(abi, n, getattr(abi, precision), 300.0, f, u, bc, k).cpu().numpy()
        res.append(np.linalg.norm(_neumann_residual(f.cpu().numpy(), out, n, walls, 1.0 / n[0], 300.0, 1.3)))
    rates = np.array(res[1:]) / np.array(res[:-1])
    assert rates.max() < 0.25, rates


@pytest.mark.parametrize("pre,post", [(1, 1), (3, 2), (1, 3), (0, 2), (4, 1)])
def test_other_sweep_counts_reach_the_same_solution(abi, pre, post):
    """sweep counts with other halos, and those the legs leave to the per-level kernels"""
    from synthetic import small_2d

    from ._util import gpu_grid, rel_err

    wl = small_2d(64, nbody=2, seed=3)
    lam = []
    for sweeps in ((2, 2), (pre, post)):
        G = gpu_grid(abi, wl, abi.MIXED)
        try:
            o = abi.solve_opts_default()
            o.tol = 1e-9
            o.mg_pre, o.mg_post = sweeps
            assert abi.solve_coupled(G, wl.UO(), opts=o).status == abi.OK
            lam.append(abi.get_forces(G, 2)[0])
        finally:
            abi.destroy_grid(G)
    assert rel_err(lam[1], lam[0]) < 1e-8
