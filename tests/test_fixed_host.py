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
    got, _ = fixed_host.cells(z[:-1], z[-1], NAN_KEYS)
    assert np.array_equal(got, np.full(NAN_KEYS.size, z.size - 2))
