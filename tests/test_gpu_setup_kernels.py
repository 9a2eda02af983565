"""Set-up kernels at the edges of their blocks: the scan behind the gather lists
(4096 entries per block, 1024 block sums per pass) through the spreading it
feeds, and the 128-row diagonal blocks of the M~ factorisation through its solve.

Tolerances.  Spreading: FP64 sums of at most N W^d products, 1e-13 N^(1/2) of the
result's norm covers their order.  Solve: an inverse formed in FP32 from a
Cholesky factor has a relative error of at most c n u kappa (Higham, Accuracy and
Stability, 2002, sec. 10 and 14; u = 2^-24), asserted with c = 10."""
import numpy as np
import pytest

from oracle import ib
from synthetic import Body, Workload, sphere_markers

from ._util import gpu_grid, oracle_problem, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def abi():
    from paper_1505_07865_gb300 import abi as a

    assert torch.cuda.is_available()
    return a


def _patch_2d(N):  # N points of a square lattice of spacing 1.5 h on a 64^2 grid
    m = int(np.ceil(np.sqrt(N)))
    p = np.stack(np.meshgrid(np.arange(m), np.arange(m)), -1).reshape(-1, 2)[:N]
    return Workload("patch", (64, 64), (1.0, 1.0), tol=1e-8,
                    bodies=[Body(np.array([0.31, 0.42]), (p - p.mean(0)) * 1.5 / 64, np.zeros(3))])


def _spheres_3d(B, N):
    rng = np.random.default_rng(B)
    return Workload("many", (64, 64, 64), (1.0, 1.0, 1.0), tol=1e-8,
                    bodies=[Body(rng.uniform(0.0, 1.0, 3), sphere_markers(0.05, N), np.zeros(6)) for _ in range(B)])


@pytest.mark.parametrize("wl", [_patch_2d(n) for n in (1, 127, 128, 129, 385)] + [_spheres_3d(220, 100)],
                         ids=["32", "4064", "4096", "4128", "12320", "4224000"])
def test_gather_lists_at_block_edges(abi, wl):
    pr = oracle_problem(wl)
    g = pr.grid
    G = gpu_grid(abi, wl, abi.MIXED)
    try:
        abi.prepare(G)
        lam = np.random.default_rng(3).standard_normal((pr.N, g.d))
        f = torch.zeros(g.d * g.ncell, dtype=torch.float64, device="cuda")
        abi.op_spread(G, torch.from_numpy(lam).cuda(), f)
        ref = np.concatenate([a.ravel() for a in ib.spread_tilde(g, pr.q, lam)])
        assert rel_err(f.cpu().numpy(), ref) < 1e-13 * max(1.0, pr.N ** 0.5)
    finally:
        abi.destroy_grid(G)


@pytest.mark.parametrize("N", [1, 12, 42, 43, 128, 129, 300])
def test_diagonal_blocks_of_the_factorisation(abi, N):
    rel = sphere_markers(0.25, N) if N > 1 else np.zeros((1, 3))
    wl = Workload("block", (64, 64, 64), (1.0, 1.0, 1.0), tol=1e-8,
                  bodies=[Body(np.array([0.5, 0.5, 0.5]), rel, np.zeros(6))])
    G = gpu_grid(abi, wl, abi.MIXED)
    try:
        abi.prepare(G)
        n = 3 * N
        Mt = torch.zeros(n * n, dtype=torch.float64, device="cuda")
        abi.op_mtilde(G, 0, Mt)
        M = Mt.cpu().numpy().reshape(n, n)
        x = np.random.default_rng(5).standard_normal(n)
        out = torch.zeros(n, dtype=torch.float64, device="cuda")
        abi.op_mtilde_solve(G, torch.from_numpy(M @ x).cuda(), out)
        assert rel_err(out.cpu().numpy(), x) < 10 * n * 2.0 ** -24 * np.linalg.cond(M)
    finally:
        abi.destroy_grid(G)
