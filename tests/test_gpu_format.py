"""What the fixed-point kernels do at the edges of their format and of their
tables, on the GPU (tests/test_fixed_host.py has the routines on the CPU)."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2012_08221_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

ALL_ONES = """
import numpy as np, torch
from paper_2012_08221_gb300 import build, synth
build.build()
from paper_2012_08221_gb300.batch import Batch
from paper_2012_08221_gb300.pdf import PDF, PDF_S_DOMAIN
for g in (synth.grid_small(), synth.grid_nnpdf()):
    p = PDF.from_grid(g)
    for n in (33, 60_001):                      # tables in global and in shared memory
        bad = torch.full((n,), -1, dtype=torch.int64, device="cuda").view(torch.float64)
        one = torch.full((n,), 0.1, dtype=torch.float64, device="cuda")
        pid = torch.full((n,), 2, dtype=torch.int32, device="cuda")
        out = torch.empty((n, 2), dtype=torch.float64, device="cuda")
        for x, q in ((bad, one * 100), (one, bad), (bad, bad)):
            assert p.xfxQ2(g.pids, x, q).isnan().all() and p.xfxQ2_pw(pid, x, q).isnan().all()
            f, a = p.xfxQ2_alphasQ2(g.pids, x, q)
            assert f.isnan().all() and bool(a.isnan().all()) == (q is bad)
            Batch([(p, 0, g.pids[:2].copy(), x, q, out)], autotune=False).run()
            assert out.isnan().all() and p.status() == PDF_S_DOMAIN
        assert p.alphasQ2(bad).isnan().all() and p.alphasQ(bad).isnan().all() and p.status() == PDF_S_DOMAIN
"""


@pytest.mark.parametrize("checked", ["0", "1"])
def test_points_of_all_ones_are_domain_errors(checked):
    """A buffer filled with 0xFF: NaN and the domain bit, and no table index out
    of range on the range-checked library."""
    r = subprocess.run([sys.executable, "-c", ALL_ONES], cwd=ROOT, capture_output=True, text=True, timeout=600,
                       env=dict(os.environ, PDFGPU_CHECKED=checked, PYTHONPATH=ROOT))
    assert r.returncode == 0, r.stderr[-3000:]


@pytest.mark.parametrize("interp", [1, 2])
def test_straight_lines_next_to_far_larger_values(interp):
    """Log-bilinear, and straight lines in a short Q subgrid: knots 2^25 above a
    cell's own on the rows and columns that it does not read.  Values and
    derivatives of the points whose own knots are the small ones (between 1 and
    2^50 the value follows the rounding of t), against the oracle."""
    from oracle.oracle import OracleGrid
    from paper_2012_08221_gb300 import build
    from paper_2012_08221_gb300.pdf import PDF
    from tests import parity
    build.build()
    rng = np.random.default_rng(31)
    x = synth.log_knots(1e-4, 1.0, 12)
    q, nq = synth.subgrid_knots([1.3, 4.0, 90.0, 500.0], [3, 3, 3])
    v = rng.uniform(1, 2, (1, q.size, x.size, 3))
    v[:, ::3] *= 2.0 ** 25                       # the first row of every subgrid; the others beside it
    if interp == 1:
        v[:, :, ::3] *= 2.0 ** 25
    g = synth.Grid(x, nq, q, np.array([-1, 1, 2], np.int32), v, np.full(q.size, 0.2), "steps")
    pdf, o = PDF.from_grid(g, interp=interp), OracleGrid.from_synth(g, interp=interp)
    n = 20_011
    xs, q2 = np.exp(rng.uniform(np.log(1e-4), 0, n)), np.exp(rng.uniform(2 * np.log(1.3), 2 * np.log(500), n))
    row = np.searchsorted(np.unique(q) ** 2, q2, side="right") - 1
    col = np.searchsorted(x, xs, side="right") - 1
    own = (row % 2 == 1) & ((col % 3 == 1) | (interp == 2))
    xs, q2 = xs[own], q2[own]
    n = xs.size
    assert n > 2000
    X, Q = torch.as_tensor(xs, device="cuda"), torch.as_tensor(q2, device="cuda")
    parity.check(pdf.xfxQ2(g.pids, X, Q).cpu().numpy(), o.xfxq2_batch(g.pids, xs, q2), o.kappa(g.pids, xs, q2))
    pid = np.full(n, 2, np.int32)
    dx, dq, _ = pdf.xfxQ2_backward(torch.as_tensor(pid, device="cuda"), X, Q,
                                   torch.ones(n, dtype=torch.float64, device="cuda"), pointwise=True)
    rdx, rdq = o.grad_pw(pid, xs, q2)
    kap = o.kappa(pid, xs, q2, pointwise=True)
    dU, dW = np.min(np.diff(np.log(x))), np.min(np.diff(2 * np.log(np.unique(q))))
    # the suite's gradient rule: 1e-9 of the value's terms over the smallest knot spacing
    for got, ref, s in ((dx, rdx, dU * xs), (dq, rdq, dW * q2)):
        assert np.all(np.abs(got.cpu().numpy() - ref) <= 1e-9 * np.maximum(np.abs(ref), 4 * kap / s))


def test_knots_uneven_on_both_axes():
    """Intervals of very different widths next to each other in x and in Q^2:
    the values at every pair of knots, next to them and in between, against
    the oracle and, at the knots, against the grid's own values."""
    from oracle.oracle import OracleGrid
    from paper_2012_08221_gb300 import build
    from paper_2012_08221_gb300.pdf import PDF
    from tests import parity
    build.build()
    rng = np.random.default_rng(41)
    steps = 2.0 ** -np.array([2, 8, 2, 15, 2, 13, 3, 5, 2, 14, 2])
    x = np.exp(np.concatenate([[0.0], np.cumsum(steps)]) - 4.0)
    w = np.concatenate([[0.0], np.cumsum(steps[::-1])])
    qa, qb = np.exp(1.0 + w / 2), np.exp(1.0 + w[-1] / 2 + w / 2)
    qb[0] = qa[-1]
    q, nq = np.concatenate([qa, qb]), np.array([qa.size, qb.size], np.int32)
    lx, lq = np.log(x)[None, :, None], 2 * np.log(q)[:, None, None]
    v = np.exp(lx * np.array([-0.4, 0.3, 0.9])) * (1 + 0.1 * lq)
    g = synth.Grid(x, nq, q, np.array([-1, 0, 1], np.int32), v[None], 0.3 / (1 + 0.1 * lq[:, 0, 0]), "uneven")
    pdf, o = PDF.from_grid(g), OracleGrid.from_synth(g)
    X, Q = (a.ravel() for a in np.meshgrid(x, q * q))
    pdf.status()
    at = pdf.xfxQ2(g.pids, torch.as_tensor(X, device="cuda"), torch.as_tensor(Q, device="cuda")).cpu().numpy()
    parity.check(at, o.xfxq2_batch(g.pids, X, Q), o.kappa(g.pids, X, Q), what="knots")
    assert np.allclose(at, v.reshape(-1, 3), rtol=1e-12, atol=0)
    k, j = rng.integers(0, x.size - 1, 20_003), rng.integers(0, q.size - 1, 20_003)
    tx, tq = (2.0 ** -rng.uniform(0, 40, (2, 20_003)))
    xs, qs = x[k] * (x[k + 1] / x[k]) ** tx, (q[j] * (q[j + 1] / q[j]) ** tq) ** 2
    xs, qs = np.clip(xs, x[0], x[-1]), np.clip(qs, q[0] ** 2, q[-1] ** 2)
    D = [torch.as_tensor(a, device="cuda") for a in (xs, qs)]
    parity.check(pdf.xfxQ2(g.pids, *D).cpu().numpy(), o.xfxq2_batch(g.pids, xs, qs), o.kappa(g.pids, xs, qs))
    parity.check(pdf.alphasQ2(D[1]).cpu().numpy(), o.alphas_batch(qs), o.alphas_kappa(qs), what="alpha_s")
    assert pdf.status() == 0


def test_knots_give_their_own_values():
    """Every knot that opens a cell returns the grid's value itself, bit for bit,
    and alpha_s likewise; with flavours that set in at a threshold and ones
    that fall away towards the next knot."""
    from paper_2012_08221_gb300 import build
    from paper_2012_08221_gb300.pdf import PDF
    build.build()
    for g in (synth.grid_small(), synth.grid_nnpdf()):
        rng = np.random.default_rng(51)
        g.values[..., 1] *= 2.0 ** rng.integers(-14, 15, g.values.shape[1:3])
        if g.n_q.size > 1:
            g.values[:, np.asarray(g.q_knots) <= 4.92, :, 2] = 0.0
        pdf = PDF.from_grid(g)
        last = np.cumsum(g.n_q) - 1                       # the last row of a subgrid opens no cell
        rows = np.setdiff1d(np.arange(g.n_rows), last)
        X, Q = (a.ravel() for a in np.meshgrid(g.x_knots[:-1], g.q_knots[rows] ** 2))
        X, Q = torch.as_tensor(X, device="cuda"), torch.as_tensor(Q, device="cuda")
        want = np.ascontiguousarray(g.values[0][rows][:, :-1].reshape(-1, g.n_flav))
        assert np.array_equal(pdf.xfxQ2(g.pids, X, Q).cpu().numpy(), want)
        q = torch.as_tensor(g.q_knots[rows] ** 2, device="cuda")
        assert np.array_equal(pdf.alphasQ2(q).cpu().numpy(), g.alphas[rows])


@pytest.mark.parametrize("k", [2, 4, 6, 8, 10, 13])
def test_values_next_to_a_small_corner(k):
    """Knots whose value is 2^-k of their neighbours': the value itself on them,
    the one in 60 digits next to them and in their cells, the same bits from the
    matrix form with few and with all columns, the pointwise form and the
    batch; derivatives with and without the tapes the same bits."""
    from paper_2012_08221_gb300 import build
    from paper_2012_08221_gb300.batch import Batch
    from paper_2012_08221_gb300.pdf import PDF
    from tests import fixed_host, parity
    build.build()
    g = synth.grid_nnpdf(seeds=(61,))
    rng = np.random.default_rng(60 + k)
    low = np.zeros(g.values.shape[1:3], bool)
    low[1::3, 1::3] = True
    g.values[...] = rng.uniform(1, 2, g.values.shape)
    g.values[:, low] *= 2.0 ** -k
    pdf = PDF.from_grid(g)
    r, c = np.nonzero(low)
    keep = (c < g.n_x - 1) & ~np.isin(r, np.cumsum(g.n_q) - 1)
    r, c = np.repeat(r[keep], 8), np.repeat(c[keep], 8)
    n = r.size
    x, q2 = g.x_knots[c].copy(), g.q_knots[r] ** 2
    tx, tq = 2.0 ** -rng.uniform(0, 40, (2, n))
    x[n // 2:] = (x * (g.x_knots[c + 1] / x) ** tx)[n // 2:]
    q2[n // 2:] = (q2 * (g.q_knots[r + 1] ** 2 / q2) ** tq)[n // 2:]
    X, Q = torch.as_tensor(x, device="cuda"), torch.as_tensor(q2, device="cuda")
    got = pdf.xfxQ2(g.pids, X, Q)
    assert np.array_equal(got[:n // 2].cpu().numpy(), g.values[0][r, c][:n // 2])
    some = np.concatenate([rng.choice(n, 100), np.arange(n // 2, n)[::n // 100]])
    for i in some:                       # (the oracle's own logarithms, to 2^-49, are not good enough here)
        s = int(np.searchsorted(np.cumsum(g.n_q), r[i], side="right"))
        rows = slice(int(np.sum(g.n_q[:s])), int(np.sum(g.n_q[:s + 1])))
        near = slice(max(c[i] - 1, 0), c[i] + 3)
        ref = fixed_host.exact(g.x_knots[near], g.q_knots[rows] ** 2, g.values[0, rows, near, 3], x[i:i + 1], q2[i:i + 1])
        parity.check(got[i, 3].item(), float(ref[0][0]), float(ref[0][1]), atol=0)
    pid = torch.as_tensor(g.pids[np.arange(n) % g.n_flav], device="cuda")
    assert torch.equal(pdf.xfxQ2_pw(pid, X, Q), got[torch.arange(n), torch.arange(n) % g.n_flav])
    assert torch.equal(pdf.xfxQ2(g.pids[4:7], X[-1001:], Q[-1001:]), got[-1001:, 4:7])
    out = torch.empty((n, 3), dtype=torch.float64, device="cuda")
    Batch([(pdf, 0, g.pids[4:7].copy(), X, Q, out)], autotune=False).run()
    assert torch.equal(out, got[:, 4:7])
    w = torch.as_tensor(rng.standard_normal(n), device="cuda")
    gv = torch.zeros(g.values.shape[1:], dtype=torch.float64, device="cuda")
    T, D, TM = pdf.new_tape(n), pdf.new_dtape(n), pdf.new_tape(n)
    pdf.xfxQ2_pw(pid, X, Q, tape=T, dtape=D)
    pdf.xfxQ2(g.pids, X, Q, tape=TM)
    a = pdf.xfxQ2_backward(pid, X, Q, w, pointwise=True, grad_values=gv, tape=T, dtape=D)[:2]
    b = pdf.xfxQ2_backward(pid, X, Q, w, pointwise=True)[:2]
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    go = w[:, None].expand(n, g.n_flav).contiguous()
    a = pdf.xfxQ2_backward(g.pids, X, Q, go, grad_values=gv, tape=TM)[:2]
    b = pdf.xfxQ2_backward(g.pids, X, Q, go)[:2]
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


@pytest.mark.parametrize("extrap", ["linear", "freeze", "error", "continuation"])
@pytest.mark.parametrize("n", [1, 32, 64, 2016, 70_016])
def test_blocks_of_points_outside_the_knots(extrap, n):
    """Runs of 32 points that all lie outside, between runs that lie inside: the
    same bits for every point as in a shuffled order, in x*f, the pointwise
    form and alpha_s; the same luminosity but for the order of its sum of 11
    pairs of values up to about 3 (11 x 2^-53 x 9 each); the same status."""
    from paper_2012_08221_gb300 import build
    from paper_2012_08221_gb300.lumi import DeviceEvents, luminosity
    from paper_2012_08221_gb300.pdf import PDF
    build.build()
    g = synth.grid_set_b()
    pdf = PDF.from_grid(g, extrap=extrap)
    rng = np.random.default_rng(70 + n)
    out = (np.arange(n) // 32) % 2 == 0
    x = np.exp(rng.uniform(np.log(1e-8), 0, n))
    q2 = np.exp(rng.uniform(2 * np.log(1.65), 2 * np.log(1e5), n))
    low = out & (np.arange(n) // 64 % 2 == 0)
    x[low] *= 1e-10
    q2[out & ~low] = np.where(rng.uniform(size=n) < 0.5, 0.3, 1e13)[out & ~low]
    perm = rng.permutation(n)
    pid = torch.as_tensor(g.pids[np.arange(n) % g.n_flav], device="cuda")
    X, Q, P = (torch.as_tensor(a, device="cuda") for a in (x, q2, perm))

    def same(a, b):
        return np.array_equal(a[P].cpu().numpy(), b.cpu().numpy(), equal_nan=True)
    pdf.status()
    a = (pdf.xfxQ2(g.pids, X, Q), pdf.xfxQ2_pw(pid, X, Q), pdf.alphasQ2(Q), *pdf.xfxQ2_alphasQ2(g.pids[:3], X, Q))
    first = pdf.status()
    b = (pdf.xfxQ2(g.pids, X[P], Q[P]), pdf.xfxQ2_pw(pid[P], X[P], Q[P]), pdf.alphasQ2(Q[P]),
         *pdf.xfxQ2_alphasQ2(g.pids[:3], X[P], Q[P]))
    assert all(same(u, w) for u, w in zip(a, b)) and first == pdf.status()
    ev = synth.events_lhc(n, seed=71)
    ev.flags[:] = np.where(out, ev.flags | 1, ev.flags & 0)
    d = DeviceEvents.from_host(ev)
    e = DeviceEvents(d.ln_tau[P], d.y[P], d.flags[P], d.ln_mu2[P], d.ln_x1[P], d.ln_s)
    (_, l1, a1), (_, l2, a2) = luminosity(pdf, d), luminosity(pdf, e)
    assert same(a1, a2)                   # (lanes share an event's pairs: the order of its sum may differ)
    assert torch.allclose(l1[P], l2, rtol=1e-12, atol=1e-13, equal_nan=True)


def test_a_grid_loads_where_only_the_fp64_table_fits():
    """Device memory for the FP64 table and the values but not for the
    fixed-point table beside them: the grid loads, leaves the rest of the
    memory alone, and gives the oracle's values; with plenty of memory the table
    is there, and freeing the grid gives it back."""
    from oracle.oracle import OracleGrid
    from paper_2012_08221_gb300 import build
    from paper_2012_08221_gb300.pdf import PDF
    from tests import parity
    build.build()
    g = synth.grid_nnpdf(seeds=tuple(range(81, 81 + 32)))
    pdf, o = PDF.from_grid(g), OracleGrid.from_synth(g)          # kernels and context loaded
    cells = (g.n_x - 1) * int(np.sum(g.n_q - 1)) * g.n_flav * g.n_members
    table = cells * 16 * 8
    del pdf
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free0 = torch.cuda.mem_get_info()[0]
    pdf = PDF.from_grid(g)
    assert 2 * table <= free0 - torch.cuda.mem_get_info()[0] < 2.2 * table
    x, q2, _ = synth.queries_nnpdf(3001, seed=82)
    X, Q = torch.as_tensor(x, device="cuda"), torch.as_tensor(q2, device="cuda")
    full = pdf.xfxQ2(g.pids, X, Q, member=5)
    del pdf
    torch.cuda.synchronize()
    assert abs(free0 - torch.cuda.mem_get_info()[0]) < 0.1 * table
    for left in (2 * table + g.values.nbytes // 3, 4 * table):
        fill = torch.empty(int(torch.cuda.mem_get_info()[0] - left) // 8, dtype=torch.float64, device="cuda")
        before = torch.cuda.mem_get_info()[0]
        pdf = PDF.from_grid(g)
        assert before - torch.cuda.mem_get_info()[0] < 1.2 * table
        got = pdf.xfxQ2(g.pids, X, Q, member=5)
        parity.check(got.cpu().numpy(), o.xfxq2_batch(g.pids, x, q2, member=5), o.kappa(g.pids, x, q2, member=5))
        parity.check(full.cpu().numpy(), o.xfxq2_batch(g.pids, x, q2, member=5), o.kappa(g.pids, x, q2, member=5))
        del pdf, fill
        torch.cuda.empty_cache()


@pytest.mark.parametrize("n", [1, 33, 3001])
def test_luminosity_with_an_unpaired_flavour(n):
    """A flavour without an antiflavour next to b quarks that set in at their
    threshold (patches that keep FP64) and events outside the knots: lum, the
    saved factors of the paired flavours, and the gradient from the saved and
    from recomputed factors, which leaves the unpaired flavour alone."""
    from oracle.oracle import OracleGrid
    from paper_2012_08221_gb300 import build
    from paper_2012_08221_gb300.lumi import DeviceEvents, luminosity, luminosity_backward
    from paper_2012_08221_gb300.pdf import PDF
    from tests import parity
    from tests.test_gpu_lumi import _event_logs
    build.build()
    full = synth.grid_nnpdf(seeds=(91,))
    v = np.concatenate([full.values, 0.7 * full.values[..., 3:4]], axis=3)
    pids = np.append(full.pids, 22).astype(np.int32)
    v[:, np.asarray(full.q_knots) <= 4.92, :, 1] = v[:, np.asarray(full.q_knots) <= 4.92, :, 11] = 0.0
    g = synth.Grid(full.x_knots, full.n_q, full.q_knots, pids, v, full.alphas, "unpaired")
    pdf, o = PDF.from_grid(g), OracleGrid.from_synth(g)
    ev = synth.events_lhc(n, seed=92, tail=0.2)
    d = DeviceEvents.from_host(ev)
    save = torch.full((n, 2, g.n_flav), float("nan"), dtype=torch.float64, device="cuda")
    L, lum, _ = luminosity(pdf, d, save_p=save)
    Lr, lumr, _ = o.lumi(ev)
    u1, u2, w = _event_logs(ev, n)
    kap, f = [], []
    for k, u in enumerate((u1, u2)):
        x, q2 = np.exp(u), np.exp(w)
        f.append(o.xfxq2_batch(pids, x, q2))
        kap.append(o.kappa(pids, x, q2))
        parity.check(save[:, k, :13].cpu().numpy(), f[k][:, :13], kap[k][:, :13], what=f"saved parton {k}")
    a = slice(0, 13)
    terms = kap[0][:, a] * np.abs(f[1][:, 12::-1]) + np.abs(f[0][:, a]) * kap[1][:, 12::-1] + \
        kap[0][:, a] * kap[1][:, 12::-1]
    parity.check(lum.cpu().numpy(), lumr, terms.sum(1), what="lum")
    ref = o.lumi_dgrid(ev)
    tol = 1e-9 * np.maximum(np.abs(ref), o.lumi_dgrid(ev, absval=True)) + 1e-300      # the suite's gradient rule
    for saved in (save, None):
        gv = torch.zeros(g.values.shape[1:], dtype=torch.float64, device="cuda")
        luminosity_backward(pdf, d, 1.0, gv, saved_p=saved)
        got = gv.cpu().numpy()
        assert np.all(np.abs(got - ref) <= tol) and not got[..., 13].any()


def test_wide_multiply_probe():
    """The rate that the x*f roofline divides by: 64 products per clock and SM
    (within a tenth on chains with operands of their own, less where all pairs
    of operands meet), at the largest clock or below it."""
    from paper_2012_08221_gb300 import build
    from paper_2012_08221_gb300.pdf import WIDE_MODES, wide_multiply_peak
    build.build()
    peak = 64 * 2.07e9 * torch.cuda.get_device_properties(0).multi_processor_count
    rate = {m: wide_multiply_peak(m) for m in WIDE_MODES}
    assert 0.5 * peak < rate["all_pairs"] <= rate["own"] <= 1.01 * peak and rate["own"] <= 1.01 * rate["shared"]
