"""The fixed-point evaluation at the edges of what it serves: cells wider and
narrower than its logarithm holds, values at the ends of the block exponent
and beyond, patches with a corner far below their largest value, zeros, short
and ragged queries, few and many columns, and queries where every other
point falls to the FP64 queue.  Every value against the oracle."""
import numpy as np
import pytest

from oracle.oracle import OracleGrid
from paper_2012_08221_gb300 import synth
from tests import parity

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# widths in ln x: 13.8 (too wide), 6.2, 0.59, 0.11, 4e-5 and 2e-5 (too narrow)
X_KNOTS = np.array([1e-9, 1e-3, 0.5, 0.9, 1 - 6e-5, 1 - 2e-5, 1.0])
# the first six flavours are one function times a power of two: inside and beyond the block exponent
SCALES = 2.0 ** np.array([0, -830, -200, -133, 83, 116, 0, 0])


@pytest.fixture(scope="module")
def odd():
    from paper_2012_08221_gb300 import build
    from paper_2012_08221_gb300.pdf import PDF
    build.build()
    rng = np.random.default_rng(81)
    q, nq = synth.subgrid_knots([1.0, 1.3, 200.0], [2, 5])
    v = rng.uniform(0.5, 2.0, (2, q.size, X_KNOTS.size, SCALES.size))
    v[..., 1:6] = v[..., :1]
    v *= SCALES
    v[:, :, 2, 6] *= 2.0 ** -20                 # corners far below the patch's other values
    v[:, :4, :, 7] = 0.0                        # a flavour that sets in at a knot
    g = synth.Grid(X_KNOTS, nq, q, np.array([-3, -2, -1, 0, 1, 2, 3, 4], np.int32), v,
                   rng.uniform(0.1, 0.4, q.size), "odd")
    return g, {e: PDF.from_grid(g, extrap=e) for e in ("linear", "freeze", "error", "continuation")}, \
        {e: OracleGrid.from_synth(g, extrap=k) for k, e in enumerate(("linear", "freeze", "error", "continuation"))}


def _points(n, outside):
    rng = np.random.default_rng(82 + n)
    k = rng.integers(0, X_KNOTS.size - 1, n)
    x = X_KNOTS[k] * (X_KNOTS[k + 1] / X_KNOTS[k]) ** rng.uniform(0, 1, n)
    x = np.clip(x, X_KNOTS[k], X_KNOTS[k + 1])
    q2 = np.exp(rng.uniform(0.0, 2 * np.log(200.0), n))
    x[::5] = X_KNOTS[k[::5]]
    if outside:
        x[1::4] *= 1e-2 / np.maximum(x[1::4], 1e-2) * 1e-9
        q2[3::4] *= np.where(q2[3::4] < 20.0, 1e-4, 1e6)
    return x, q2


# (no power laws carried far outside this grid's widest cells: there the
# oracle and the FP64 path differ by the amplified rounding of the exponent)
@pytest.mark.parametrize("extrap,n,outside",
                         [(e, n, o) for e in ("linear", "freeze", "error", "continuation")
                          for n, o in ((1, False), (31, True), (33, False), (1000, True), (20_001, True),
                                       (90_007, False)) if not (o and e == "continuation")])
def test_values_at_the_format_limits(odd, extrap, n, outside):
    g, pdfs, oracles = odd
    pdf, o = pdfs[extrap], oracles[extrap]
    x, q2 = _points(n, outside)
    X, Q = torch.as_tensor(x, device="cuda"), torch.as_tensor(q2, device="cuda")
    pdf.status()
    got = pdf.xfxQ2(g.pids, X, Q, member=1).cpu().numpy()
    ref, kap = o.xfxq2_batch(g.pids, x, q2, member=1), o.kappa(g.pids, x, q2, member=1)
    # the scaled flavours are judged on the unscaled function (not under the
    # continuation, whose threshold of 1e-3 is no power of two's)
    for a in range(g.n_flav):
        b = a if a > 5 or extrap == "continuation" else 0
        parity.check(got[:, a] * (SCALES[b] / SCALES[a]), ref[:, b], kap[:, b], what=f"{extrap} flavour {a}")
    assert pdf.status() == (2 if extrap == "error" and outside else 0)
    # one flavour per point, alpha_s beside, other column counts: the same bits
    pid = torch.as_tensor(g.pids[np.arange(n) % g.n_flav], device="cuda")
    pw = pdf.xfxQ2_pw(pid, X, Q, member=1).cpu().numpy()
    assert np.array_equal(pw, got[np.arange(n), np.arange(n) % g.n_flav], equal_nan=True)
    out, a_s = pdf.xfxQ2_alphasQ2(g.pids, X, Q, member=1)
    assert np.array_equal(out.cpu().numpy(), got, equal_nan=True)
    assert np.array_equal(a_s.cpu().numpy(), pdf.alphasQ2(Q).cpu().numpy(), equal_nan=True)
    for cols in ([4], [6, 1, 9], list(range(8)) * 2 + [0], list(range(8)) * 8):
        pids = np.array([g.pids[c] if c < 8 else 40 for c in cols], np.int32)      # 40: absent
        few = pdf.xfxQ2(pids, X, Q, member=1).cpu().numpy()
        for k, c in enumerate(cols):
            want = got[:, c] if c < 8 else np.where(np.isnan(got[:, 0]), np.nan, 0.0)
            assert np.array_equal(few[:, k], want, equal_nan=True)


@pytest.mark.parametrize("n", [1, 31, 33, 2000, 60_001])
def test_luminosity_with_flavours_that_set_in_at_a_threshold(n):
    """Events (5 % of them outside the knots) on a grid whose b quarks are zero
    up to their threshold knot, so that the patches above it keep FP64, with
    an unpaired flavour: lum and alpha_s per event, the saved partner
    factors, and the VEGAS sums of the same luminosity."""
    from oracle.oracle import vegas_sums
    from paper_2012_08221_gb300.lumi import DeviceEvents, luminosity
    from paper_2012_08221_gb300.pdf import PDF
    from paper_2012_08221_gb300.vegas import VegasLumi
    from tests.test_gpu_lumi import _as_kappa, _event_logs, _lum_kappa
    g = synth.grid_nnpdf(seeds=(83, 84))
    rows = np.asarray(g.q_knots) <= 4.92
    g.values[:, rows, :, 1] = g.values[:, rows, :, 11] = 0.0
    pdf, o = PDF.from_grid(g), OracleGrid.from_synth(g)
    ev = synth.events_lhc(n, seed=85)
    d = DeviceEvents.from_host(ev)
    save = torch.full((n, 2, g.n_flav), 7.0, dtype=torch.float64, device="cuda")
    L, lum, a_s = luminosity(pdf, d, member=1, save_p=save)
    L2, lum2, _ = luminosity(pdf, d, member=1)
    _, lumr, asr = o.lumi(ev, member=1)
    kap = _lum_kappa(g, o, ev, n, member=1)
    parity.check(lum.cpu().numpy(), lumr, kap, what="lum")
    parity.check(a_s.cpu().numpy(), asr, _as_kappa(o, ev, n), what="alpha_s")
    assert torch.equal(lum, lum2) and abs(L.item() - L2.item()) <= 1e-12 * kap.sum() / n
    u1, u2, w = _event_logs(ev, n)
    for k, u in enumerate((u1, u2)):            # exp() of the logarithms: the parity rule's scale covers its rounding
        x, q2 = np.exp(u), np.exp(w)
        parity.check(save[:, k].cpu().numpy(), o.xfxq2_batch(g.pids, x, q2, member=1),
                     o.kappa(g.pids, x, q2, member=1), what=f"saved parton {k}")
    v = np.random.default_rng(86).uniform(0, 1, (n, 2))
    vg = VegasLumi(pdf, np.log(1e-6), 2 * np.log(13000.0), n_bins=20, member=1)
    _, _, s = vg.iteration(torch.as_tensor(v, device="cuda"), refine=False)
    ref = vegas_sums(o, 1, np.log(1e-6), 2 * np.log(13000.0), np.tile(np.linspace(0, 1, 21), (2, 1)), v)
    assert np.all(np.abs(s - ref) <= 1e-11 * np.abs(ref) + 1e-300)


@pytest.mark.parametrize("n", [1, 31, 33, 2000, 30_001])
def test_derivatives_of_the_matrix_and_the_pointwise_form(n):
    """dL/dx and dL/dQ^2 of one column through the matrix form (quads of lanes)
    and the pointwise form with the derivative tape: each the same bits with
    the tapes and without, with points on knots, outside the grid and in
    patches that keep FP64; both against the oracle's derivative."""
    from paper_2012_08221_gb300.pdf import PDF
    g = synth.grid_nnpdf(seeds=(87, 88))
    g.values[:, np.asarray(g.q_knots) <= 4.92, :, 11] = 0.0
    pdf, o = PDF.from_grid(g), OracleGrid.from_synth(g)
    x, q2, _ = synth.queries_nnpdf(n, seed=89)
    x[::7], q2[3::7] = g.x_knots[np.arange(x[::7].size) % 190], 4.92 ** 2
    x[5::11], q2[6::11] = 3e-11, 1e12
    X, Q = torch.as_tensor(x, device="cuda"), torch.as_tensor(q2, device="cuda")
    w = torch.as_tensor(np.random.default_rng(90).standard_normal(n), device="cuda")
    for pid in (5, -2):
        col = np.array([pid], np.int32)
        pids = torch.full((n,), pid, dtype=torch.int32, device="cuda")
        gv = torch.zeros(g.values.shape[1:], dtype=torch.float64, device="cuda")
        T, D, TM = pdf.new_tape(n), pdf.new_dtape(n), pdf.new_tape(n)
        pdf.xfxQ2_pw(pids, X, Q, member=1, tape=T, dtape=D)
        pdf.xfxQ2(col, X, Q, member=1, tape=TM)
        a = pdf.xfxQ2_backward(pids, X, Q, w, member=1, pointwise=True, grad_values=gv, tape=T, dtape=D)[:2]
        for b in (pdf.xfxQ2_backward(pids, X, Q, w, member=1, pointwise=True, grad_values=gv, tape=T)[:2],
                  pdf.xfxQ2_backward(pids, X, Q, w, member=1, pointwise=True)[:2]):
            assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
        mat = pdf.xfxQ2_backward(col, X, Q, w[:, None], member=1, grad_values=gv, tape=TM)[:2]
        for b in (pdf.xfxQ2_backward(col, X, Q, w[:, None], member=1, grad_values=gv)[:2],
                  pdf.xfxQ2_backward(col, X, Q, w[:, None], member=1)[:2]):
            assert torch.equal(mat[0], b[0]) and torch.equal(mat[1], b[1])
        pn = np.full(n, pid, np.int32)
        rdx, rdq = o.grad_pw(pn, x, q2, member=1)
        kap = o.kappa(pn, x, q2, member=1, pointwise=True)
        U, W = np.log(g.x_knots), np.log(g.q_knots ** 2)
        dW = np.diff(W)
        wn = w.cpu().numpy()
        # the suite's gradient rule: 1e-9 of the value's terms over the smallest knot spacing
        sx, sq = np.min(np.diff(U)) * x, np.min(dW[dW > 0]) * q2
        for got, ref, s in ((a[0], rdx, sx), (a[1], rdq, sq), (mat[0], rdx, sx), (mat[1], rdq, sq)):
            err = np.abs(got.cpu().numpy() - wn * ref)
            assert np.all(err <= 1e-9 * np.maximum(np.abs(wn * ref), np.abs(wn) * 4 * kap / s) + 1e-300)


@pytest.mark.parametrize("power", [0, 1, 9, 10, 11, 12, 60])
def test_continuation_between_values_of_any_ratio(power):
    """The power law from edge values whose ratio stays inside the logarithm's
    format, at its limit (2^10) and beyond.  Two Q knots, the upper row 2^power
    times the lower: the edge values come out of the patch to full precision
    (with more rows the patch's own sums lose the smaller one)."""
    from paper_2012_08221_gb300.pdf import PDF
    x = np.array([1e-4, 1e-3, 1e-2, 0.1, 0.4])
    q, nq = synth.subgrid_knots([2.0, 60.0], [2])
    rng = np.random.default_rng(91 + power)
    v = rng.uniform(1.0, 1.9, (1, 2, 5, 2))
    v[:, 1] *= 2.0 ** power
    a = np.array([0.3, 0.3 * 2.0 ** power])
    g = synth.Grid(x, nq, q, np.array([1, 2], np.int32), v, a, "ratio")
    pdf, o = PDF.from_grid(g, extrap="continuation"), OracleGrid.from_synth(g, extrap=3)
    n = 4003
    xs = np.minimum(np.exp(rng.uniform(np.log(3e-5), 0.0, n)), 1.0)
    q2 = np.exp(rng.uniform(2 * np.log(1.2), 2 * np.log(100.0), n))
    X, Q = torch.as_tensor(xs, device="cuda"), torch.as_tensor(q2, device="cuda")
    parity.check(pdf.xfxQ2(g.pids, X, Q).cpu().numpy(), o.xfxq2_batch(g.pids, xs, q2), o.kappa(g.pids, xs, q2),
                 what=f"ratio 2^{power}")
    parity.check(pdf.alphasQ2(Q).cpu().numpy(), o.alphas_batch(q2), o.alphas_kappa(q2), what="alpha_s")
