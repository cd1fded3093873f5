"""The outflow mass-flux correction, summed by many blocks, on planes of every kind of remainder."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1812_01178_gb300 import binding as B
from paper_1812_01178_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# faces: fewer than the 1024 partial sums, as many, one row more, one pass of 16 each, a little more, several
@pytest.mark.parametrize("ny, nz", [(20, 8), (64, 16), (41, 32), (128, 128), (129, 128), (200, 256)])
def test_outflow_shift(ny, nz):
    case, u, v, w, p, bl = I.boundary_layer(16, ny, nz)
    rng = np.random.default_rng(7)
    u = u.copy()
    u[:, :, 0] += rng.standard_normal((nz, ny))
    bl = dict(bl, u_out=bl["u_out"] + rng.standard_normal((nz, ny)))
    s = B.Solver(case, u, v, w, p, bl=bl)
    s.make_divergence_free()  # the shift, then the projection (which leaves the plane alone)
    s.sync()
    got = s.boundary()["u_out"]
    s.close()
    dy = np.diff(np.asarray(case.yf))
    terms = (u[:, :, 0] - bl["u_out"]) * dy
    scale = 1.0 / (nz * (case.yf[-1] - case.yf[0]))  # dz / (Ly Lz)
    corr = math.fsum(terms.ravel()) * scale
    # a partial sum of ceil(n / 1024) terms, ten levels of the tree, the roundings of a term, of the
    # factor and of the shift itself
    eps = 2.0 ** -53
    tol = eps * ((ny * nz // 1024 + 1) + 10 + 6) * np.abs(terms).sum() * scale
    want = bl["u_out"] + corr
    assert (np.abs(got - want) <= tol + 2 * eps * np.abs(want)).all(), np.abs(got - want).max()
