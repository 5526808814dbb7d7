"""The host/device routines of the fixed-point evaluation, on the CPU (the
same source that the kernels inline, built by tests/fixed_host.py)."""
import numpy as np
import pytest

from paper_2012_08221_gb300 import synth
from tests import fixed_host

NAN_KEYS = np.array([0x7FF0000000000000, 0x7FF8000000000000, 0x8000000000000000, 0xFFF8000000000000,
                     0xFFFFFFFF00000000, 0xFFFFFFFFFFFFFFFE, 0xFFFFFFFFFFFFFFFF], np.uint64)


@pytest.mark.parametrize("knots", [[0.1, 1.0], [1e-4, 0.5, 1.0], [1e-9, 1e-3, 0.5, 0.9, 1 - 6e-5, 1 - 2e-5, 1.0],
                                   synth.log_knots(1e-9, 1.0, 196),
                                   np.concatenate([synth.log_knots(1e-5, 0.5, 9), 0.5 + 2.0 ** -40 * np.arange(1, 12),
                                                   [1.0]]),
                                   # steps from 2^-12 to 2^-46: no bucket width fits, binary search
                                   np.concatenate([[1e-6, 0.5], 0.5 + np.cumsum(2.0 ** -np.arange(46.0, 2.0, -2.0)),
                                                   [1.0]])])
def test_search_gives_a_cell_for_every_bit_pattern(knots):
    """Points are searched before their domain is tested, so infinities,
    negative numbers and NaNs (a buffer of all ones among them) must give a cell
    of the table too; keys of the range give theirs."""
    z = np.asarray(knots, np.float64)
    rng = np.random.default_rng(3)
    x = np.concatenate([z, np.nextafter(z, 0), np.nextafter(z, 2), np.exp(rng.uniform(np.log(z[0]) - 5, 1, 2000))])
    got, _ = fixed_host.cells(z[:-1], z[-1], x.view(np.uint64))
    assert np.array_equal(got, np.clip(np.searchsorted(z[:-1], x, side="right") - 1, 0, z.size - 2))
    assert np.array_equal(fixed_host.cells(z[:-1], z[-1], np.arange(3, dtype=np.uint64))[0], np.zeros(3))
    got, _ = fixed_host.cells(z[:-1], z[-1], NAN_KEYS)
    assert np.array_equal(got, np.full(NAN_KEYS.size, z.size - 2))


def _points(x, q2, cell, n, rng):
    """Points of cell (i, j) in both axes: at its lower knots, near them (down to
    2^-30 of the cell) on one axis and on both, and anywhere."""
    i, j = cell
    tx, tq = rng.uniform(0, 1, n), rng.uniform(0, 1, n)
    tx[::3] = 2.0 ** -rng.uniform(0, 30, tx[::3].size)
    tq[::2] = 2.0 ** -rng.uniform(0, 30, tq[::2].size)
    px = np.clip(x[i] * (x[i + 1] / x[i]) ** tx, x[i], np.nextafter(x[i + 1], 0))
    pq = np.clip(q2[j] * (q2[j + 1] / q2[j]) ** tq, q2[j], np.nextafter(q2[j + 1], 0))
    px[:8], pq[4:12] = x[i], q2[j]
    return px, pq


@pytest.mark.parametrize("x_linear,q_linear", [(True, True), (False, True)])
@pytest.mark.parametrize("power", [0, 10, 20, 40, 60, 200])
def test_straight_lines_next_to_far_larger_values(power, x_linear, q_linear):
    """Linear axes read the two knots of their interval only: neighbours 2^power
    larger leave the cell's value and derivatives alone.  Every coefficient is
    at most 2^3 here (values in [1, 2)), so that the fixed-point error, 2^-57 of
    it in the value and four times that in a derivative, and the rounding to a
    double stay below 2^-52 and 2^-50 of the weighted values."""
    rng = np.random.default_rng(200 + power)
    x, q2 = np.exp(-2 + 0.1 * np.arange(4)), np.exp(3 + 0.1 * np.arange(4))
    v = rng.uniform(1, 2, (4, 4))
    v[[0, 3]] *= 2.0 ** power
    if x_linear:
        v[:, [0, 3]] *= 2.0 ** power
    px, pq = _points(x, q2, (1, 1), 60, rng)
    got, t = fixed_host.evaluate(x, q2, v, px, pq, x_linear, q_linear)
    ref = fixed_host.exact(x, q2, v, px, pq, t, x_linear, q_linear)
    kap = np.array([float(r[1]) for r in ref])
    assert np.all(np.isfinite(got))
    for col, k, tol in ((0, 0, 2.0 ** -52), (2, 2, 2.0 ** -50), (3, 3, 2.0 ** -50)):
        err = fixed_host.error(got[:, col], [r[k] for r in ref])
        assert np.all(err <= tol * np.maximum(kap, 1.0)), (col, np.max(err / kap))


def test_non_finite_neighbours_of_a_straight_line_keep_fp64():
    """The FP64 form multiplies them by its zero weights, which gives NaN; the
    fixed-point form does not serve such a patch."""
    x, q2 = np.exp(-2 + 0.1 * np.arange(4)), np.exp(3 + 0.1 * np.arange(4))
    for bad in (np.inf, np.nan):
        v = np.ones((4, 4))
        v[0, 1] = bad
        got, _ = fixed_host.evaluate(x, q2, v, x[1:2], q2[1:2], True, True)
        assert np.isnan(got[0, 0]) and np.isnan(got[0, 1])


def _uneven(r, rng):
    """Knots whose second interval is 2^r times its lower neighbour."""
    d = rng.uniform(0.02, 0.4)
    return -2 + np.array([-d * 2.0 ** -r, 0.0, d, d * rng.uniform(1.3, 4.0)])


@pytest.mark.parametrize("r", [0, 3, 5, 6, 8, 10, 12, 14, 15])
def test_uneven_cells_on_both_axes(r):
    """Smooth positive values on a cell that is 2^r times its lower neighbour on
    both axes, at its knots and inside.  Where fixed point serves, what the
    build leaves is at most 2^(E - 53), E at most 1 above the corner's exponent
    for values that vary by less than 2 over the cell, and the corner at least
    half of 2^that: 2^-51 of the values, and 2^-50 with the evaluation's and
    the rounding's share."""
    rng = np.random.default_rng(300 + r)
    served = 0
    for _ in range(6):
        u, w = _uneven(r, rng), 5 + _uneven(r, rng)
        a, b = rng.uniform(-0.5, 0.5), rng.uniform(-0.02, 0.1)
        v = np.exp(a * u)[None] * (1 + b * w)[:, None]
        x, q2 = np.exp(u), np.exp(w)
        px, pq = _points(x, q2, (1, 1), 60, rng)
        got, t = fixed_host.evaluate(x, q2, v, px, pq)
        ref = fixed_host.exact(x, q2, v, px, pq, t)
        kap = np.array([float(k[1]) for k in ref])
        ok = np.isfinite(got[:, 0])
        served += ok.sum()
        err = fixed_host.error(got[:, 0], [k[0] for k in ref])
        assert np.all(err[ok] <= 2.0 ** -50 * kap[ok]), np.max(err[ok] / kap[ok])
    assert served == 360 if r <= 4 else True          # ordinary cells stay in fixed point


@pytest.mark.parametrize("what", ["corner", "column", "row"])
@pytest.mark.parametrize("k", [0, 1, 2, 3, 4, 6, 8, 10, 12, 14])
def test_values_small_at_the_lower_edges(k, what):
    """Cells whose corner, left column or lower row is 2^-k of the rest.  Where
    fixed point serves: the knot's value itself at the corner; next to it within
    2^-52 of the value where fixed point serves the edges too (off by 2^(E - 56)
    at most, the corner at least 2^(E - 2), and the rounding adds 2^-53); and
    over the whole cell no larger an error against the exact value of the
    argument, on the scale of the weighted values, than the FP64 form."""
    rng = np.random.default_rng(400 + k)
    fixed, fp64, served = [], [], 0
    for _ in range(8):
        u = np.concatenate([[-5.0], -5 + np.cumsum(0.1 * 7.0 ** rng.uniform(-0.5, 0.5, 3))])
        w = np.concatenate([[2.0], 2 + np.cumsum(0.2 * 7.0 ** rng.uniform(-0.5, 0.5, 3))])
        x, q2 = np.exp(u), np.exp(w)
        v = rng.uniform(1, 2, (4, 4)) * rng.choice([-1, 1])
        v[(1, 1) if what == "corner" else np.s_[:, 1] if what == "column" else np.s_[1]] *= 2.0 ** -k
        px, pq = _points(x, q2, (1, 1), 60, rng)
        px[:20] = np.clip(x[1] * (1 + rng.uniform(0, 1e-9, 20)), x[1], None)
        pq[:20] = np.clip(q2[1] * (1 + rng.uniform(0, 1e-9, 20)), q2[1], None)
        px[0], pq[0] = x[1], q2[1]
        got, t = fixed_host.evaluate(x, q2, v, px, pq)
        ok = np.isfinite(got[:, 0])
        if ok[0]:
            assert got[0, 0] == v[1, 1]
        near = fixed_host.exact(x, q2, v, px[:20], pq[:20], t)
        err = fixed_host.error(got[:20, 0], [r[0] for r in near])
        assert np.all(err[ok[:20]] <= 2.0 ** -52 * abs(v[1, 1]))
        ref = fixed_host.exact(x, q2, v, px, pq)
        kap = np.array([float(r[1]) for r in ref])
        fixed.append((fixed_host.error(got[:, 0], [r[0] for r in ref]) / kap)[ok])
        fp64.append((fixed_host.error(got[:, 4], [r[0] for r in ref]) / kap)[ok])
        served += ok.sum()
    fixed, fp64 = np.concatenate(fixed), np.concatenate(fp64)
    if k <= 4:
        assert served >= 100                             # away from the edges at least
    if fixed.size:
        assert np.max(fixed) <= np.max(fp64)


def test_alpha_s_cubics():
    """The centred cubics of alpha_s where they serve: exact at the lower knots,
    and within 2^-52 of the terms' size in between, on even and uneven knots."""
    rng = np.random.default_rng(500)
    for r in (0, 4, 8, 12):
        w = np.cumsum(np.concatenate([[1.0], 0.3 * 2.0 ** -rng.permutation([r, 0, 1, 0, r, 0])]))
        a = 1.3 / (1 + 0.6 * w) + 0.01 * rng.uniform(0, 1, w.size)
        q2 = np.exp(w)
        p = np.concatenate([q2[:-1], np.exp(rng.uniform(w[0], w[-1], 80))])
        got, t = fixed_host.alphas(q2, a, p)
        ref = fixed_host.exact(q2, np.array([1.0, 2.0]), np.vstack([a, a]), p, np.ones(p.size),
                               np.column_stack([t, np.zeros_like(t)]))
        kap = np.array([float(k[1]) for k in ref])
        ok = np.isfinite(got)
        assert ok.sum() >= (got.size if r == 0 else got.size // 2)
        assert np.array_equal(got[:w.size - 1][ok[:w.size - 1]], a[:-1][ok[:w.size - 1]])
        assert np.all(fixed_host.error(got, [k[0] for k in ref])[ok] <= 2.0 ** -52 * kap[ok])


@pytest.mark.parametrize("j", [3, 5, 7, 8, 9, 10, 11, 13])
@pytest.mark.parametrize("axis", ["x", "q"])
def test_narrow_cells_next_to_one(j, axis):
    """Knots 2^-j / 5 apart up to x = 1 (or from Q^2 = 1 on): there the FP64
    logarithm is accurate to its own size, the fixed-point one to 2^-59, and a
    narrow cell magnifies both.  Where fixed point serves, its error against the
    exact value of the argument is no larger than that of FP64."""
    rng = np.random.default_rng(600 + j)
    h = 2.0 ** -j
    near = 1 - h * np.array([1.0, 0.82, 0.58, 0.4, 0.19, 0.0]) if axis == "x" else 1 + h * np.arange(6) / 5
    far = np.exp(np.arange(5) * 0.3 + (2 if axis == "x" else -3))
    x, q2 = (near, far) if axis == "x" else (far, near)
    fixed, fp64 = [], []
    for smooth in (False, True):
        v = rng.uniform(1, 2, (q2.size, x.size))
        if smooth:
            v = (2 - x)[None] ** 3 * (1 + 0.1 * np.log(q2))[:, None]
        px, pq = rng.uniform(x[0], x[-1], 250), rng.uniform(q2[0], q2[-1], 250)
        got, _ = fixed_host.evaluate(x, q2, v, px, pq)
        ref = fixed_host.exact(x, q2, v, px, pq)
        kap = np.array([float(r[1]) for r in ref])
        fixed.append(fixed_host.error(got[:, 0], [r[0] for r in ref]) / kap)
        fp64.append(fixed_host.error(got[:, 4], [r[0] for r in ref]) / kap)
    fixed, fp64 = np.concatenate(fixed), np.concatenate(fp64)
    served = np.isfinite(fixed)
    assert served.all() if j <= 3 else True
    if served.any():
        assert np.max(fixed[served]) <= np.max(fp64)


@pytest.mark.parametrize("seed", range(8))
def test_steep_falls_on_uneven_cells(seed):
    """A function that falls by orders of magnitude over coarse and uneven cells,
    (1 - x)^b up to x = 1, at points near both ends of the cells: the matrices'
    row sums, the stencil's range and the cancellation towards the far knot all
    meet.  Where fixed point serves, its error against the exact value of the
    argument, on the scale of the weighted values, is no larger than FP64's: root
    mean square against root mean square, and the largest within twice the
    largest (of 480 points each, a few of which lie where both cancel)."""
    rng = np.random.default_rng(700 + seed)
    fixed, fp64 = [], []
    for _ in range(4):
        u = -np.cumsum(np.exp(rng.uniform(-3, 2, 5)))[::-1]
        x = np.append(np.exp(u - 0.01), 1.0)
        q2 = np.exp(3 + np.cumsum(0.2 * np.exp(rng.uniform(-1, 1, 5))))
        v = x[None] ** rng.uniform(-0.5, 1) * np.maximum(1 - x, 0)[None] ** rng.uniform(2, 6) * \
            (1 + rng.uniform(-0.05, 0.1) * np.log(q2))[:, None]
        n = 120
        k, j = rng.integers(0, x.size - 1, n), rng.integers(0, q2.size - 1, n)
        t, s = 2.0 ** -rng.uniform(0, 10, (2, n))
        t[::2], s[::4] = 1 - t[::2], 1 - s[::4]
        px = np.clip(x[k] * (x[k + 1] / x[k]) ** t, x[k], np.nextafter(x[k + 1], 0))
        pq = np.clip(q2[j] * (q2[j + 1] / q2[j]) ** s, q2[j], np.nextafter(q2[j + 1], 0))
        got, _ = fixed_host.evaluate(x, q2, v, px, pq)
        ref = fixed_host.exact(x, q2, v, px, pq)
        kap = np.array([float(r[1]) for r in ref])
        ok = np.isfinite(got[:, 0]) & (kap > 0)
        fixed.append((fixed_host.error(got[:, 0], [r[0] for r in ref])[ok] / kap[ok]))
        fp64.append((fixed_host.error(got[:, 4], [r[0] for r in ref])[ok] / kap[ok]))
    fixed, fp64 = np.concatenate(fixed), np.concatenate(fp64)
    assert fixed.size > 50 and np.max(fixed) <= 2 * np.max(fp64), (np.max(fixed), np.max(fp64))
    assert np.mean(fixed ** 2) <= np.mean(fp64 ** 2)


@pytest.mark.parametrize("j", [3, 5, 6, 7])
def test_falls_to_zero_in_narrow_cells_next_to_one(j):
    """(1 - x)^4 over knots 2^-j / 5 apart up to x = 1, where the value follows the
    coordinate's relative accuracy: fixed point, where it serves, is no further
    from the exact value of the argument than FP64 (root mean square and largest
    error on the scale of the weighted values)."""
    rng = np.random.default_rng(800 + j)
    x = 1 - 2.0 ** -j * np.array([1.0, 0.82, 0.58, 0.4, 0.19, 0.0])
    q2 = np.exp(2 + 0.3 * np.arange(5))
    v = np.maximum(1 - x, 0)[None] ** 4 * (1 + 0.1 * np.log(q2))[:, None]
    px, pq = rng.uniform(x[0], x[-1], 400), rng.uniform(q2[0], q2[-1], 400)
    got, _ = fixed_host.evaluate(x, q2, v, px, pq)
    ref = fixed_host.exact(x, q2, v, px, pq)
    kap = np.array([float(r[1]) for r in ref])
    ok = np.isfinite(got[:, 0]) & (kap > 0)
    if ok.any():
        fixed = fixed_host.error(got[:, 0], [r[0] for r in ref])[ok] / kap[ok]
        fp64 = fixed_host.error(got[:, 4], [r[0] for r in ref])[ok] / kap[ok]
        assert np.max(fixed) <= np.max(fp64) and np.mean(fixed ** 2) <= np.mean(fp64 ** 2)
