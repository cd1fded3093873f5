"""The FP64 right-hand side in fixed point on tiles of unequal values: which arithmetic a cell takes shows
in its last bits, since a row next to a plane that holds a NaN is formed in FP64 arithmetic."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ns_oracle as O
from paper_1812_01178_gb300 import binding as B
from paper_1812_01178_gb300 import inputs as I

pytestmark = pytest.mark.gpu

OUT = (B.NS_BUF_RU, B.NS_BUF_RV, B.NS_BUF_RW, B.NS_BUF_NU, B.NS_BUF_NV, B.NS_BUF_NW)


def _rhs(case, f, k=0):
    s = B.Solver(case, *f)
    s.rhs(k)
    s.sync()
    out = [s.buffer(b).cpu().numpy().copy() for b in OUT]
    s.close()
    return out


def _in_fp64(case, f):
    """The same with every row in FP64 arithmetic, without the cells that read the NaN: one cell of each
    32 x 8 tile of u's every third row spoils the rows next to it."""
    g = [a.copy() for a in f]
    g[0][::8, ::3, ::32] = np.nan
    return _rhs(case, g)


@pytest.mark.parametrize("zero", ["", "w", "vw", "uv", "u"])
def test_zero_components_take_the_fixed_point_path(zero):
    """Two-dimensional and parallel flows, and a component at rest: no plane of zeros sends a row to FP64
    arithmetic.  Both agree to the rounding of either (1e-13 of the field's largest)."""
    case, u, v, w, p = I.small_channel(64, 23, 16, seed=11)
    f = [u, v, w, p]
    for q in zero:
        f["uvw".index(q)] = np.zeros_like(f["uvw".index(q)])
    got, ref = _rhs(case, f), _in_fp64(case, f)
    for q, (a, b) in enumerate(zip(got, ref)):
        fin = np.isfinite(b)
        assert fin.mean() > 0.5
        if not b[fin].any():
            assert not a.any(), q
            continue
        assert np.abs(a[fin] - b[fin]).max() <= 1e-13 * np.abs(b[fin]).max(), q
        # every row of cells (v: of inner faces) of a component that moves differs somewhere, so no row of
        # `got` was formed in FP64
        rows = (fin & (a != b)).any(axis=(0, 2))
        if f[q % 3].any():
            assert (rows[1:-1] if a.shape[1] > case.ny else rows).all(), (q, np.flatnonzero(~rows))


def _near(f, rows):
    """Largest |f| within a cell in x and z and two rows, on rows 0 .. rows - 1."""
    m = np.zeros((f.shape[0], rows, f.shape[2]))
    m[:, :f.shape[1]] = np.abs(f)
    for axis in (0, 2):
        m = np.maximum(m, np.maximum(np.roll(m, 1, axis), np.roll(m, -1, axis)))
    p = np.pad(m, ((0, 0), (2, 2), (0, 0)))
    return np.max([p[:, q:q + rows] for q in range(5)], axis=0)


@pytest.mark.parametrize("pulse, tol", [
    # v and w: their values keep 53 bits of the largest of a cell and its neighbours in x and z, which is at
    # least 2^-9 of the largest of the tile's three planes; a convective sum is then off by at most four units
    # of 2^-60 2^11 of its largest term (u is of one size): 2^-47, and the oracle's own roundings
    ("vw", 1e-14),
    # all three: products of two such values, 2^-60 2^(9 + 9 + 2 + 2)
    ("uvw", 2.0 ** -38),
])
@pytest.mark.parametrize("size", [(64, 23, 16), (48, 9, 24)])
def test_quiet_cells_beside_a_pulse(size, pulse, tol):
    """Single cells 1e8 times the rest of their tile: the sums of the others keep their digits, each against
    the largest terms of its own neighbourhood."""
    case, u, v, w, p = I.small_channel(*size, seed=13)
    rng = np.random.default_rng(size[0])
    f = [u, v, w]
    for q in pulse:
        a = f["uvw".index(q)] = 1e-8 * rng.standard_normal(f["uvw".index(q)].shape)
        for i in range(0, size[0], 16):  # two in every tile, on any row and column
            for k in range(0, size[2], 8):
                a[k + rng.integers(8), 1 + rng.integers(size[1] - 2), i + rng.integers(8)] = 1.0
    f[1][:, [0, -1]] = 0.0
    p = 0.0 * p
    g = O.Grid.from_case(case)
    got = _rhs(case, f + [p])
    r, n = O.rhs(g, *f, p, None, 0, case.dt, case.re, 0.0)
    gam, vis = case.dt * O.RK3_GAMMA[0], case.dt * O.RK3_ALPHA[0] / case.re
    rows = case.ny + 1
    mu, mv, mw = (_near(q, rows) for q in f)
    h = np.diff(case.yf).min()
    rate = 2 * (mu / g.dx + mv / h + mw / g.dz)
    lap = 4 / g.dx ** 2 + 4 / g.dz ** 2 + 4 / h ** 2
    fx = case.dt * O.RK3_ALPHA[0] * case.fx
    for q, m in enumerate((mu, mv, mw)):
        size_n, size_r = gam * rate * m, (gam * rate + vis * lap) * m + (fx if q == 0 else 0.0)
        c = got[q].shape[1]
        assert (np.abs(got[q] - r[q] - (fx if q == 0 else 0.0)) <= tol * size_r[:, :c]).all(), q
        assert (np.abs(got[3 + q] + gam * n[q]) <= tol * size_n[:, :c]).all(), q
