"""The plain mixed schedule's own sub-cycle loop (every k in one) against the
binned schedule, bit for bit, on warps of mixed k: every order, both field-time
readings, electrons that cross nodes either way or none, and at the window's
ends; and the device memory that a plain context takes."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2102_10983_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2102_10983_gb300 import native  # noqa: E402


@pytest.mark.parametrize("ratio", [0.125, 0.99, 4.0])
@pytest.mark.parametrize("order", [1, 2, 3, 4, 5])
def test_plain_has_the_binned_bits(ratio, order):
    n, width, dt, steps = 12001, 64, W.DT75, 3
    rng = np.random.Generator(np.random.PCG64(int(100 * ratio) + order))
    shape = np.sin(np.arange(width) * rng.uniform(0.3, 1.0)) * 40.0
    E, B = (np.array([shape * (1 + 0.1 * l) * s for l in range(order + steps)]) for s in (0.7, 1.0))
    x = rng.uniform(1.0, width - 1.0, n)
    edge = rng.random(n) < 0.1
    x[edge] = rng.choice((1.0, width - 2.0), edge.sum()) + rng.uniform(-0.6, 0.6, edge.sum())
    p = rng.normal(0, 1, (3, n)) * np.exp(rng.uniform(-2, 3, n))
    out = []
    for sched in (native.PIC_SCHED_PLAIN, native.PIC_SCHED_BINNED):
        it = native.Integrator(dt, dt / ratio, 0.01, order=order, precision=native.PIC_MIXED, schedule=sched,
                               field_time=order % 2, capacity=n, window=width, ring_levels=order + steps + 1)
        it.pic_particles_write(x * (dt / ratio), *p)
        for l in range(order + steps):
            it.pic_fields_upload(l - order, 0, E[l], B[l])
        st, _ = it.pic_push_step(0, steps, ok=(native.PIC_OK, native.PIC_ERANGE, native.PIC_EKMAX))
        out.append((it.read_numpy(), st.as_dict()))
        it.close()
    for a, b in zip(out[0][0], out[1][0]):
        np.testing.assert_array_equal(a, b)
    assert out[0][1] == out[1][1]
    assert min(out[0][1]["k_hist"][:5]) > 0 and out[0][1]["out_of_window"] > 0


@pytest.mark.parametrize("order,tables", [(1, 0), (3, 1), (5, 0)])
def test_plain_holds_only_the_tables_it_reads(order, tables):
    width, ring = 1 << 20, order + 2
    native.Integrator(W.DT75, W.DT75, 0.01, order=order, precision=native.PIC_MIXED, capacity=16).close()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    it = native.Integrator(W.DT75, W.DT75, 0.01, order=order, precision=native.PIC_MIXED, capacity=16, window=width,
                           ring_levels=ring)
    used = free - torch.cuda.mem_get_info()[0]
    it.close()
    # node fields, feature nodes, the two mirrored rings, staging (2^22 doubles), tables
    need = width * (16 + 8 + 2 * 2 * ring * 4 + tables * 8 * (order + 1)) + (1 << 25)
    assert used < need + width * 4 * (order + 1)  # less than half a table more
