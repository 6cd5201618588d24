"""The coupled loop by its routes, against the oracle bit for bit: small ensembles
in one launch (a warp per electron, up to three per SM), electrons fewer than
the grid's entries (levels gathered), as many (node fields); and what a large
grid costs a small ensemble."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2102_10983_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2102_10983_gb300 import native  # noqa: E402
from test_gpu_sc1d_paths import test_sc1d_unsorted_electrons_and_odd_charges as _both  # noqa: E402


@pytest.mark.parametrize("n,cells,qm,order", [
    (2, 16, -1.0, 2), (700, 300, -0.4, 4), (3 * 152, 300, -1.0, 3), (3 * 152 + 1, 600, -1.0, 3),
    (1500, 4000, -1.0, 1), (1500, 4000, 0.3, 2), (1500, 4000, 1.0, 4), (1500, 4000, -1.0, 5),
    (3004, 3000, -1.0, 3), (3005, 3000, -1.0, 3)])
def test_routes(n, cells, qm, order):
    _both(n, cells, qm, order, "wide")


def _loop(n, cells):
    g = native.Sc1d(W.DT75, W.DT75 / 0.99, cells, psi_max=1e30, capacity=n)
    z = torch.zeros(n, dtype=torch.float64, device="cuda")
    g.particles_write(z + 30.0 * W.DT75, z, z, z, z)
    f = torch.zeros(cells + 5, dtype=torch.float64, device="cuda")
    for l in range(4):
        g.fields_write(l - 3, f, f, f)
    return g


def test_small_ensembles_take_one_launch():
    g = _loop(100, 200)
    before = g.launches()
    g.step(0, 4)
    assert g.launches() - before == 4 * 2  # the push, the fields
    g.close()


def test_a_large_grid_does_not_slow_a_small_ensemble():
    """2,000 electrons on 2^22 cells: the push adds little to the field solve (a
    pass over the grid's entries would take as long as that)."""
    ms = {}
    for n in (0, 2000):
        g = _loop(n, 1 << 22)
        t = []
        for q in range(9):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            g.step(4 * q, 4, want_stats=False)
            b.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(b) / 4)
        ms[n] = sorted(t)[4]
        g.close()
    assert ms[2000] < 1.3 * ms[0] + 0.06, ms
