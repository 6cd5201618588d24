"""A captured FP64 step replayed: every replay counts and groups its sub-cycled
electrons anew.  Bit for bit as the same calls made one by one."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2102_10983_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2102_10983_gb300 import native  # noqa: E402


@pytest.mark.parametrize("n,steps", [(40, 1), (5000, 1), (5000, 3)])
def test_replayed_steps(n, steps):
    p, width, dx = 3, 64, W.DT75 / 0.99
    rng = np.random.Generator(np.random.PCG64(n + steps))
    E, B = rng.uniform(-30.0, 30.0, (2, p + steps, width))
    x = rng.uniform(20.0, 40.0, n) * dx
    mom = rng.normal(0.0, 2.0, (3, n))
    stream = torch.cuda.Stream()
    out = []
    for captured in (False, True):
        it = native.Integrator(W.DT75, dx, 0.01, order=p, k_max=7, precision=native.PIC_FP64, capacity=n,
                               window=width, ring_levels=p + steps, stream=stream)
        it.pic_particles_write(x, *mom)
        for r in range(p + steps):
            it.pic_fields_upload(r - p, 0, E[r], B[r])
        stream.synchronize()
        if captured:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                it.pic_push_step(0, steps, want_stats=False)
            for _ in range(4):
                graph.replay()
            torch.cuda.synchronize()
        else:
            for _ in range(4):
                it.pic_push_step(0, steps, want_stats=False)
        out.append(it.read_numpy())
        st = it.pic_stats_read()
        assert sum(st.k_hist[1:]) > 0
        out[-1] = list(out[-1]) + [np.array(st.k_hist)]
        it.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
