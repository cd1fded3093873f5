"""The fixed-point forms of the FP64 path: values outside their range take FP64 arithmetic.

The Poisson solve is linear, and scaling its input by a power of two scales every FP64 operation
exactly, so a solve whose values lie near an end of the binary64 range (general path) must agree with
the same solve at ordinary magnitudes (fixed point) to the rounding of either."""
import numpy as np
import pytest

from paper_1812_01178_gb300 import binding as B
from paper_1812_01178_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# stage sequences: radix 4 alone, radix 2 first, radix 3 last, both; tiles of 2 to 16 columns
SIZES = [(64, 5, 16), (32, 6, 8), (24, 5, 72), (72, 4, 24), (16, 4, 1024), (1024, 4, 8), (144, 5, 48)]


def _phi(case, u, v, w, p):
    s = B.Solver(case, u, v, w, p)
    s.poisson(-1)
    s.sync()
    phi = s.buffer(B.NS_BUF_PHI).cpu().numpy().copy()
    s.close()
    return phi


def _inputs(size, plate):
    if plate:  # (the outflow planes stay zero)
        case, u, v, w, p, bl = I.boundary_layer(*size)
        return case, u, v, w, p
    return I.small_channel(*size, seed=5)


@pytest.mark.parametrize("plate", [False, True])
@pytest.mark.parametrize("size", SIZES)
def test_poisson_at_the_ends_of_the_range(size, plate):
    case, u, v, w, p = _inputs(size, plate)
    ref = _phi(case, u, v, w, p)
    for e in (-940, 925):
        f = 2.0 ** e
        got = _phi(case, u * f, v * f, w * f, p) / f
        # two roundings of about 3 eps log2(n) a transform, amplified by the y solves like any FP64 rounding
        assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max(), (e, np.abs(got - ref).max())


@pytest.mark.parametrize("size", SIZES[:3])
def test_poisson_of_zero_and_of_non_finite_fields(size):
    case, u, v, w, p = I.small_channel(*size, seed=5)
    z = np.zeros_like
    assert np.array_equal(_phi(case, z(u), z(v), z(w), p), z(p))
    for bad in (np.nan, np.inf):
        u2 = u.copy()
        u2[1, 2, 3] = bad
        assert np.isnan(_phi(case, u2, v, w, p)).any()
