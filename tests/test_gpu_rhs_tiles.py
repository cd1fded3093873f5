"""The FP64 right-hand side in fixed point on tiles of unequal values: which arithmetic a cell takes shows
in its last bits, since a row next to a plane that holds a NaN is formed in FP64 arithmetic."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

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
