"""The periodic FP64 product with the system matrix forms its stencil sums in
64-bit integers scaled to the largest value of a sum; exponents near the ends of
the range, infinities and NaN take the plain formula.  Checked against the
stencil in extended precision (numpy longdouble) at value ranges where the
scaling, the cut-off bits and the switch between the two can go wrong.

Tolerance: per sum of at most 12 terms, 2^-58 of the largest term per cut-off
and one rounding to 53 bits, then three roundings of the products and sums of
kappa h^-2, the pressure difference and their total: below 8 eps of the sum of
the terms' magnitudes, row by row.
"""
import numpy as np
import pytest

from synthetic import small_2d, small_3d

from ._util import gpu_grid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


def _fields(kind, d, shape, rng):
    x = rng.standard_normal((d + 1,) + shape)
    if kind == "wide":        # neighbours up to 2^400 apart
        x *= 2.0 ** rng.integers(-200, 200, x.shape)
    elif kind == "smooth":    # sums that cancel
        x = 1.0 + 1e-9 * x
    elif kind == "holes":     # zeros and single spikes among them
        x *= rng.uniform(size=x.shape) < 0.2
    elif kind == "tiny":      # around the smallest normal numbers
        x *= 2.0 ** rng.integers(-1060, -1000, x.shape)
    elif kind == "huge":
        x *= 2.0 ** rng.integers(990, 1004, x.shape)
    return x


def _product(x, d, eta, h):
    """rows and the sum of the magnitudes of their terms, in extended precision"""
    x = x.astype(np.longdouble)
    kh2, ih = np.longdouble(eta) / (np.longdouble(h) * np.longdouble(h)), 1 / np.longdouble(h)
    p, rows, mags = x[d], [], []
    div, dmag = 0.0, 0.0
    for a in range(d):
        u, ax = x[a], d - 1 - a
        lap, lmag = -2 * d * u, 2 * d * np.abs(u)
        for b in range(d):
            for s in (1, -1):
                n = np.roll(u, s, d - 1 - b)
                lap, lmag = lap + n, lmag + np.abs(n)
        pm = np.roll(p, 1, ax)
        rows.append(-kh2 * lap + (p - pm) * ih)
        mags.append(kh2 * lmag + (np.abs(p) + np.abs(pm)) * ih)
        up = np.roll(u, -1, ax)
        div, dmag = div + (up - u), dmag + np.abs(up) + np.abs(u)
    return np.stack(rows + [-div * ih]), np.stack(mags + [dmag * ih])


@pytest.mark.parametrize("kind", ["plain", "wide", "smooth", "holes", "tiny", "huge"])
@pytest.mark.parametrize("dim", [2, 3])
def test_rows_to_rounding(dim, kind):
    from paper_1505_07865_gb300 import abi

    wl = small_2d(34, seed=3) if dim == 2 else small_3d(12, seed=4)
    G = gpu_grid(abi, wl, abi.FP64)
    try:
        abi.prepare(G)
        h = wl.L[0] / wl.n[0]
        shape = tuple(wl.n[::-1])
        x = _fields(kind, dim, shape, np.random.default_rng(8))
        xt = torch.zeros(abi.sizes(G)[0], dtype=torch.float64, device="cuda")
        xt[:x.size] = torch.as_tensor(x.ravel(), device="cuda")  # no marker forces
        y = torch.empty_like(xt)
        abi.apply_system(G, xt, y)
        got = y[:x.size].cpu().numpy().reshape(x.shape)
    finally:
        abi.destroy_grid(G)
    ref, mag = _product(x, dim, wl.eta, h)
    assert np.all(np.isfinite(got))
    assert np.all(np.abs(got - ref) <= 8 * EPS * mag + 4 * np.finfo(np.float64).tiny)


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_non_finite_values_reach_the_rows_that_use_them(value):
    from paper_1505_07865_gb300 import abi

    wl = small_3d(12, seed=4)
    G = gpu_grid(abi, wl, abi.FP64)
    try:
        abi.prepare(G)
        n = int(np.prod(wl.n))
        xt = torch.ones(abi.sizes(G)[0], dtype=torch.float64, device="cuda")
        xt[4 * n:] = 0.0
        xt[n + 5 + 12 * (6 + 12 * 7)] = value  # v_1 at cell (5, 6, 7)
        y = torch.empty_like(xt)
        abi.apply_system(G, xt, y)
        bad = ~np.isfinite(y[:4 * n].cpu().numpy().reshape(4, 12, 12, 12))
    finally:
        abi.destroy_grid(G)
    want = np.zeros_like(bad)
    for dz, dy, dx in [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]:
        want[1, 7 + dz, 6 + dy, 5 + dx] = True
    want[3, 7, 6, 5] = want[3, 7, 5, 5] = True  # the two cells that share the face
    assert np.array_equal(bad, want)


def test_an_infinite_coefficient_stays_infinite():
    """eta h^-2 = 1e310 overflows: no row of it may come out as a number (the scale of the
    integer sums is formed by adding exponents, which means something for normal numbers only)"""
    from paper_1505_07865_gb300 import abi

    n, h = 34, 1e-10
    G = abi.create_grid(2, (n, n), (n * h, n * h), eta=1e290, precision=abi.FP64)
    try:
        bid = abi.add_body(G, [0.5 * n * h] * 2)
        abi.set_markers(G, bid, np.array([[2.0 * h, 0.0], [-2.0 * h, 0.0]]))
        abi.prepare(G)
        xt = torch.zeros(abi.sizes(G)[0], dtype=torch.float64, device="cuda")
        xt[:2 * n * n] = torch.as_tensor(np.random.default_rng(9).standard_normal(2 * n * n), device="cuda")
        y = torch.empty_like(xt)
        abi.apply_system(G, xt, y)
        assert not torch.isfinite(y[:2 * n * n]).any()
    finally:
        abi.destroy_grid(G)
