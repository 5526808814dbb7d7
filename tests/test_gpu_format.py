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
