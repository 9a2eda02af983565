"""Which 2-D levels run their legs in one launch: the line lies at 450000 cells (all
stacked fields together) in FP64 and 1250000 in FP32 between walls; periodic FP32
levels have none.  A level beyond it runs one half sweep per launch, so it has a
restriction launch of its own in the event profile, which a leg does not have.

On periodic grids the FP64 result is also compared with the V-cycle of the per-level
kernels, which apply the same formulas (association of two sums aside): 1e-13 of
the largest value after a cycle, 1e-5 for FP32.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def abi():
    from paper_1505_07865_gb300 import abi as a

    assert torch.cuda.is_available()
    return a


def _grid(abi, n, walls, precision):
    bc = []
    for a in range(2):
        bc += [abi.NOSLIP if (walls >> a) & 1 else abi.PERIODIC] * 2
    return abi.create_grid(2, n, [m / n[0] for m in n], bc=bc, precision=getattr(abi, precision))


def _restrictions(abi, call):
    abi.profile_enable(True)
    try:
        abi.profile_reset()
        call()
        return abi.profile_read().get("mg_residual_restrict", (0,))[0]
    finally:
        abi.profile_enable(False)


@pytest.mark.parametrize("precision,walls,n,beyond", [
    ("FP64", 0, (704, 640), 1), ("FP64", 0, (640, 640), 0), ("FP64", 0, (1024, 1024), 1), ("FP64", 0, (2048, 1024), 2),
    ("FP64", 3, (704, 704), 1), ("FP64", 1, (448, 448), 0), ("MIXED", 0, (2048, 2048), 0),
    ("MIXED", 3, (1024, 1024), 0), ("MIXED", 2, (1536, 1024), 1)])
def test_levels_beyond_the_line(abi, precision, walls, n, beyond):
    G = _grid(abi, n, walls, precision)
    try:
        g = torch.Generator(device="cuda").manual_seed(4)
        f = torch.randn(n[0] * n[1], dtype=torch.float64, device="cuda", generator=g)
        u = torch.randn(n[0] * n[1], dtype=torch.float64, device="cuda", generator=g)
        out = u.clone()
        assert _restrictions(abi, lambda: abi.op_vcycle(G, 300.0, 1.3, f, out, 1)) == beyond
    finally:
        abi.destroy_grid(G)
    if walls == 0 and n[0] * n[1] <= 720000:  # (larger ones exceed the other entry's scratch)
        abi.op_vcycle_noalloc(2, n, [m / n[0] for m in n], 300.0, 1.3, f, u, 1)
        assert float((out - u).abs().max()) <= (1e-13 if precision == "FP64" else 1e-5) * float(u.abs().max())


@pytest.mark.parametrize("precision,n,beyond", [("FP64", (480, 480), 1), ("FP64", (448, 448), 0), ("MIXED", (1024, 1024), 0)])
def test_stacked_fields_count_together(abi, precision, n, beyond):
    """P_S: a V-cycle of two velocity components (480^2 is beyond the line) and one of the pressure (not)"""
    G = _grid(abi, n, 0, precision)
    try:
        r = torch.randn(3 * n[0] * n[1], dtype=torch.float64, device="cuda")
        z = torch.empty_like(r)
        assert _restrictions(abi, lambda: abi.op_stokes_pc(G, r, z)) == beyond
    finally:
        abi.destroy_grid(G)
