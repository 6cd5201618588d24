"""Deferred particles several steps behind the stream, read from the node tables
of the last steps and, further back, from the levels: bit for bit the plain
schedule, whatever number of tables the window's size leaves room for, from a
negative first step on, and on both sides of the length at which a stream item
takes a second tile."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2102_10983_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2102_10983_gb300 import native  # noqa: E402


# window cells (16, 8 and 2 tables of order 3), particles, first step
@pytest.mark.parametrize("width,n,first", [(64, 5001, -7), (1 << 20, 3000, 0), (1 << 22, 1, 3),
                                           (1 << 22, 2000, -30), (64, 3_300_017, 5)])
def test_lagging_particles_equal_plain(width, n, first):
    order, steps, dt = 3, 24 if n < 1 << 20 else 6, W.DT75
    dx = dt / 0.5
    rng = np.random.Generator(np.random.PCG64(width % 1000 + n))
    shape = np.zeros(width)
    shape[:64] = np.sin(np.arange(64) * 0.4) * 30.0
    x = rng.uniform(20.0, 44.0, n) * dx
    p = rng.normal(0, 1, (3, n)) * np.exp(rng.uniform(-2, 3, n))
    out = []
    for sched, budget in ((native.PIC_SCHED_PLAIN, 0), (native.PIC_SCHED_BINNED, 5)):
        it = native.Integrator(dt, dx, 0.01, order=order, precision=native.PIC_MIXED, schedule=sched,
                               capacity=n, window=width, ring_levels=order + 1 + steps,
                               heavy_budget=budget)
        it.pic_particles_write(x, *p)
        for l in range(order + steps):
            at = first - order + l
            f = shape * (1 + 0.02 * l)
            it.pic_fields_upload(at, 0, 0.7 * f, f)
        it.pic_push_step(first, steps, ok=(native.PIC_OK, native.PIC_ERANGE, native.PIC_EKMAX))
        out.append(it.read_numpy())
        it.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
    assert n == 1 or ((out[0][4] & 7) >= 3).any()
