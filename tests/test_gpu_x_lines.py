"""The FP64 x sweep line by line: every line alike, and every entry to the rounding of its own terms.

The rows are those of a diagonally dominant M-matrix, whose inverse has no negative entry: the FP64
sweep's error in a row is a few roundings of (A^-1 |d|) at that row, however large the line is elsewhere.
The bound of 1e-14 is 90 roundings: three a row of either recurrence (rows further away enter with the
powers of the decay), those of the factors and of the interface solve."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import ns_oracle as O
from paper_1812_01178_gb300 import binding as B
from paper_1812_01178_gb300 import inputs as I

pytestmark = pytest.mark.gpu

BUFS = (B.NS_BUF_RU, B.NS_BUF_RV, B.NS_BUF_RW)


def _pdd(d, r, M):
    """Cyclic solve of -r x_{i-1} + (1 + 2r) x_i - r x_{i+1} = d_i in extended precision by the sweep's own
    method: partitions of M rows, spikes, 2 x 2 interfaces.  Its sums have no cancellation beyond d's own."""
    L = np.longdouble
    r = L(r)
    x = np.asarray(d, dtype=L).reshape(*np.shape(d)[:-1], -1, M)
    piv = np.empty(M, dtype=L)
    piv[0] = 1 + 2 * r
    for e in range(1, M):
        piv[e] = 1 + 2 * r - r * r / piv[e - 1]

    def block(t):
        t = t.copy()
        for e in range(1, M):
            t[..., e] += r / piv[e - 1] * t[..., e - 1]
        t[..., M - 1] /= piv[M - 1]
        for e in range(M - 2, -1, -1):
            t[..., e] = (t[..., e] + r * t[..., e + 1]) / piv[e]
        return t

    x = block(x)
    v = block(np.eye(M, dtype=L)[0] * r)  # minus the spike of x^{(r-1)}_m; that of x^{(r+1)}_1 is its mirror image
    g0, g1 = x[..., -1], np.roll(x[..., 0], -1, -1)
    det = 1 - v[0] * v[0]
    y0, y1 = (g0 + v[0] * g1) / det, (g1 + v[0] * g0) / det
    x = x + v * np.roll(y0, 1, -1)[..., None] + v[::-1] * y1[..., None]
    return x.reshape(np.shape(d))


def _solver(nx, r, M, plate=False):
    """A solver whose x rows couple by r = beta / dx^2 in sub-step 0, in partitions of M rows (PDD)."""
    case, u, v, w, p = I.small_channel(nx, 5, 8, seed=3)
    case.dt, case.re = 1.0, O.RK3_ALPHA[0] / (2 * r * (case.lx / nx) ** 2)
    s = B.Solver(case, u, v, w, p)
    s.set_partition(nx // M, B.NS_PART_PDD)
    assert s.partition()[:2] == (nx // M, B.NS_PART_PDD)
    return s


def _sweep(s, lines):
    """x sweep of the given u, v and w lines (arrays of [lines, nx])."""
    for b, a in zip(BUFS, lines):
        t = s.buffer(b)
        t.copy_(torch.as_tensor(a.reshape(t.shape)).to(t.device))
    s.adi(0, 0)
    s.sync()
    return [s.buffer(b).cpu().numpy().reshape(-1, s.case.nx).copy() for b in BUFS]


def _live(s):
    """Lines the sweep solves: all but v's wall rows."""
    ny, nz = s.case.ny, s.case.nz
    inner = np.ones((nz, ny + 1), bool)
    inner[:, [0, ny]] = False
    return [np.ones(nz * ny, bool), inner.ravel(), np.ones(nz * ny, bool)]


@pytest.mark.parametrize("nx, M", [(64, 4), (256, 8), (256, 16), (1024, 32)])
def test_equal_lines_give_equal_results(nx, M):
    s = _solver(nx, 0.03, M)
    line = np.random.default_rng(nx).standard_normal(nx)
    got = _sweep(s, [np.tile(line, (len(q), 1)) for q in _live(s)])
    first = got[0][0]
    for g, live in zip(got, _live(s)):
        assert (g[live] == first).all()
    s.close()


@pytest.mark.parametrize("nx, M", [(64, 8), (256, 16)])
def test_small_entries_beside_a_large_one(nx, M):
    r = 0.03
    s = _solver(nx, r, M)
    rng = np.random.default_rng(nx + 1)
    lines = [rng.standard_normal((len(q), nx)) for q in _live(s)]
    for a in lines:
        a[np.arange(len(a)), rng.integers(0, nx, len(a))] = 2.0 ** 40
    got = _sweep(s, lines)
    for g, a, live in zip(got, lines, _live(s)):
        bound = _pdd(np.abs(a[live]), r, M)
        assert (np.abs(g[live] - _pdd(a[live], r, M)) <= 1e-14 * bound).all()
    s.close()


@pytest.mark.parametrize("nx, M", [(768, 24), (1024, 32), (2048, 64), (4096, 128)])
def test_long_lines_far_from_their_sources(nx, M):
    """Zero lines but for one row: the solution falls off through the neighbouring partition, by the decay
    of the rows to 1e-40 and below, and keeps its digits there (down to 1e-280: short of underflow).  Four
    roundings a row between: the factor's pivot and quotient, the spike's product and the sweep's."""
    r = 0.03
    s = _solver(nx, r, M)
    lines = [np.zeros((len(q), nx)) for q in _live(s)]
    at = 5 * M + M - 1  # the last row of a partition
    for a in lines:
        a[:, at] = 1.0
    got = _sweep(s, lines)
    want = _pdd(lines[0][0], r, M)
    near = np.flatnonzero(want > 1e-280)
    near = near[(near >= 4 * M) & (near < 7 * M)]  # the partition of the source and its neighbours
    tol = 1e-14 + 4 * 2.0 ** -53 * np.abs(near - at)
    for g, live in zip(got, _live(s)):
        assert (np.abs(g[live][:, near] - want[near]) <= tol * want[near]).all()
    s.close()


@pytest.mark.parametrize("nx, M", [(768, 24), (1024, 32)])
def test_long_lines_of_uneven_size(nx, M):
    """Entries that change by orders of magnitude from row to row, zeros, and an infinity or a NaN that stays
    in the partitions next to it."""
    r = 0.03
    s = _solver(nx, r, M)
    rng = np.random.default_rng(nx + 2)
    lines = [rng.standard_normal((len(q), nx)) * 2.0 ** rng.integers(-30, 30, (len(q), nx)) for q in _live(s)]
    for a in lines:
        a[rng.random(a.shape) < 0.1] = 0.0
    got = _sweep(s, lines)
    for g, a, live in zip(got, lines, _live(s)):
        assert (np.abs(g[live] - _pdd(a[live], r, M)) <= 1e-14 * _pdd(np.abs(a[live]), r, M)).all()
    for bad in (np.inf, np.nan):
        spoilt = [a.copy() for a in lines]
        for a in spoilt:
            a[:, 3 * M + 1] = bad
        for g, h, live in zip(_sweep(s, spoilt), got, _live(s)):
            assert not np.isfinite(g[live][:, 2 * M:5 * M]).any()
            assert (g[live][:, 6 * M:] == h[live][:, 6 * M:]).all()
    s.close()
