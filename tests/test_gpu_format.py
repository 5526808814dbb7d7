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
    """Log-bilinear, and straight lines in a short Q subgrid: knots 2^40 above a
    cell's own on the rows and columns that it does not read.  Values against
    the oracle, the luminosity's and the derivatives' patches with them."""
    from oracle.oracle import OracleGrid
    from paper_2012_08221_gb300 import build
    from paper_2012_08221_gb300.pdf import PDF
    from tests import parity
    build.build()
    rng = np.random.default_rng(31)
    x = synth.log_knots(1e-4, 1.0, 12)
    q, nq = synth.subgrid_knots([1.3, 4.0, 90.0, 500.0], [3, 3, 3])
    v = rng.uniform(1, 2, (1, q.size, x.size, 3))
    v[:, ::3] *= 2.0 ** 40                       # the first row of every subgrid; the others beside it
    if interp == 1:
        v[:, :, ::3] *= 2.0 ** 40
    g = synth.Grid(x, nq, q, np.array([-1, 1, 2], np.int32), v, np.full(q.size, 0.2), "steps")
    pdf, o = PDF.from_grid(g, interp=interp), OracleGrid.from_synth(g, interp=interp)
    n = 20_011
    xs, q2 = np.exp(rng.uniform(np.log(1e-4), 0, n)), np.exp(rng.uniform(2 * np.log(1.3), 2 * np.log(500), n))
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
    steps = 2.0 ** -np.array([2, 8, 2, 10, 3, 13, 3, 5, 2, 12, 2])
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
