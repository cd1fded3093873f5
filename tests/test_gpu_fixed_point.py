"""The fixed-point forms of the FP64 path: values outside their range take FP64 arithmetic.

The Poisson solve is linear, and scaling its input by a power of two scales every FP64 operation
exactly, so a solve whose values lie near an end of the binary64 range (general path) must agree with
the same solve at ordinary magnitudes (fixed point) to the rounding of either."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ns_oracle as O
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


def _rhs_all(s, k):
    s.rhs(k)
    s.sync()
    return [s.buffer(b).cpu().numpy().copy() for b in (B.NS_BUF_RU, B.NS_BUF_RV, B.NS_BUF_RW, B.NS_BUF_NU,
                                                       B.NS_BUF_NV, B.NS_BUF_NW)]


def _rhs_oracle(case, fields, bl):
    u, v, w, p = fields
    g = O.Grid.from_case(case)
    with np.errstate(all="ignore"):
        if bl is not None:
            r, n = O.rhs_bl(g, u, v, w, p, None, bl, 0, case.dt, case.re, case.fx)
        else:
            r, n = O.rhs(g, u, v, w, p, None, 0, case.dt, case.re, case.fx)
        return list(r) + [-case.dt * O.RK3_GAMMA[0] * q for q in n]


def _rhs_case(size, plate):
    if plate:
        case, u, v, w, p, bl = I.boundary_layer(*size, amp=0.05, seed=3, re=200.0)
        return case, [u, v, w, p], bl
    case, u, v, w, p = I.small_channel(*size, seed=5)
    return case, [u, v, w, p], None


# partial tiles in x (24, 48, 72) and z (8, 24), chunks of rows, single tiles, rows past several chunks
RHS_SIZES = [(8, 5, 8), (24, 7, 16), (48, 6, 24), (72, 13, 8), (32, 4, 32), (96, 70, 48)]


@pytest.mark.parametrize("plate", [False, True])
@pytest.mark.parametrize("size", RHS_SIZES)
def test_rhs_tiles_and_rows_of_unequal_size(size, plate):
    """The fixed-point right-hand side on every kind of partial tile, with fields whose size changes by
    1e12 over the rows and components 1e8 apart: row by row within the rounding of FP64 arithmetic on
    the largest values the row reads (1e-12, as for the whole fields elsewhere)."""
    case, f, bl = _rhs_case(size, plate)
    ny = size[1]
    row = 10.0 ** np.linspace(-9, 3, ny)
    rowf = 10.0 ** np.linspace(-9, 3, ny + 1)
    f[0] = f[0] * row[None, :, None]
    f[1] = f[1] * rowf[None, :, None] * 1e-8
    f[2] = f[2] * row[None, :, None] * 1e-4
    f[3] = f[3] * row[None, :, None]
    if bl is not None:
        bl = dict(bl, u_out=f[0][:, :, -1].copy(), v_in=bl["v_in"] * rowf * 1e-8, v_out=f[1][:, :, -1].copy(),
                  w_in=bl["w_in"] * row * 1e-4, w_out=f[2][:, :, -1].copy())
    ref = _rhs_oracle(case, f, bl)
    s = B.Solver(case, *f, bl=bl)
    got = _rhs_all(s, 0)
    s.close()
    for q, (a, b) in enumerate(zip(got, ref)):
        m = np.abs(b).max(axis=(0, 2))
        near = np.maximum(m, np.maximum(np.r_[m[1:], 0.0], np.r_[0.0, m[:-1]]))
        assert (np.abs(a - b).max(axis=(0, 2)) <= 1e-12 * near + 1e-300).all(), q


@pytest.mark.parametrize("plate", [False, True])
@pytest.mark.parametrize("size", RHS_SIZES)
def test_rhs_outside_the_fixed_point_range(size, plate):
    """Rows next to values outside the range: planes below 2^-895 and, at one cell, an infinity or a
    NaN.  Cells that do not read it keep their values, those that do become non-finite where the
    oracle's do."""
    case, f, bl = _rhs_case(size, plate)
    f[1] = f[1] * 1e-290
    f[2][:, ::2] *= 1e-285
    if bl is not None:
        bl = dict(bl, v_in=bl["v_in"] * 1e-290, v_out=bl["v_out"] * 1e-290)
        for q in ("w_in", "w_out"):
            bl[q] = bl[q].copy()
            bl[q][:, ::2] *= 1e-285
    for bad in (None, np.nan, np.inf):
        g = [a.copy() for a in f]
        if bad is not None:
            g[0][2, 2, 3] = bad
        ref = _rhs_oracle(case, g, bl)
        s = B.Solver(case, *g, bl=bl)
        got = _rhs_all(s, 0)
        s.close()
        for q, (a, b) in enumerate(zip(got, ref)):
            fin = np.isfinite(b)
            if bad is not None:
                assert not np.isfinite(a[~fin]).any(), q
                fin[1:4, 1:4, 2:5] = False
            scale = max(np.abs(b[fin]).max(), 1e-300)
            assert np.abs(a[fin] - b[fin]).max() <= 1e-12 * scale, q


@pytest.mark.parametrize("nx", [8, 24, 48, 64, 96, 144, 192, 256, 384, 512, 1024])
@pytest.mark.parametrize("plate", [False, True])
def test_x_lines_of_any_size(nx, plate):
    """Lines solved in fixed point and in FP64 side by side, each scaled on its own: lines scaled by
    powers of two (also out of the fixed-point range) give the scaled solution to the rounding of the
    sweep, a line of zeros stays zero, and a NaN stays in its line."""
    case, f, bl = _rhs_case((nx, 5, 16), plate)
    rng = np.random.default_rng(nx)
    s = B.Solver(case, *f, bl=bl)
    bufs = [s.buffer(b) for b in (B.NS_BUF_RU, B.NS_BUF_RV, B.NS_BUF_RW)]
    rows = [b.shape[0] * b.shape[1] for b in bufs]
    base = [rng.standard_normal((n, nx)) for n in rows]
    for b, a in zip(bufs, base):
        b.copy_(torch.as_tensor(a.reshape(b.shape)).to(b.device))
    s.adi(0, 0)
    s.sync()
    ref = [b.cpu().numpy().reshape(-1, nx).copy() for b in bufs]
    e = [rng.choice([-940, -300, -7, 0, 11, 300, 920], n) for n in rows]
    zero = [rng.random(n) < 0.1 for n in rows]
    bad = [rng.random(n) < 0.1 for n in rows]
    for b, a, ex, z, x in zip(bufs, base, e, zero, bad):
        t = np.ldexp(a, ex[:, None]) * ~z[:, None]
        t[x, nx // 2] = np.nan
        b.copy_(torch.as_tensor(t.reshape(b.shape)).to(b.device))
    s.adi(0, 0)
    s.sync()
    for q, (b, r, ex, z, x) in enumerate(zip(bufs, ref, e, zero, bad)):
        got = b.cpu().numpy().reshape(-1, nx)
        walls = np.zeros(b.shape[:2], bool)
        if q == 1:  # v lines on the walls are not solved
            walls[:, 0] = walls[:, -1] = True
        live = ~walls.reshape(-1)
        assert np.isnan(got[live & x]).any(axis=1).all()
        ok = live & ~x
        want = np.where(z[ok, None], 0.0, r[ok])
        have = np.ldexp(got[ok], -ex[ok, None])
        # a dozen roundings of the line's largest value either way
        assert (np.abs(have - want).max(axis=1) <= 1e-14 * np.maximum(np.abs(want).max(axis=1), 0.0)).all(), q
    s.close()
