"""The FP64 push by its routes, against the oracle bit for bit: with and without
its node fields (a window with more nodes than electrons gathers the levels),
small ensembles in one launch; and what a large window costs a small ensemble."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2102_10983_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2102_10983_gb300 import native  # noqa: E402

OK = (native.PIC_OK, native.PIC_ERANGE, native.PIC_EKMAX)


def _both(n, width, order, qm=-1.0, k_max=3, work=False, field_time=0, steps=2):
    rng = np.random.Generator(np.random.PCG64(n + width + order))
    dt = W.DT75
    dx = dt / 0.99
    i0 = np.arange(order + steps, dtype=np.int64) - 3  # a window that moves on each level
    amp = np.exp(rng.uniform(np.log(1e-3), np.log(300.0), width)) * rng.choice((-1.0, 0.0, 1.0), width, p=(.45, .1, .45))
    E, B = (amp * rng.uniform(0.5, 1.5, (order + steps, width)) for _ in range(2))
    x = rng.uniform(-4.0, width + 4.0, n) * dx  # some outside the window
    px, py, pz = rng.normal(0.0, 2.0, (3, n))
    status = rng.integers(0, 4, n).astype(np.uint8)
    status[rng.random(n) < 0.02] |= native.PIC_STATUS_LOST
    prm = oracle.Params(dt=dt, dx=dx, psi_max=0.01, order=order, k_max=k_max, qm=qm, field_time=field_time)
    ref = oracle.Particles(x, px, py, pz, status)
    wk = np.zeros(n) if work else None
    ost = oracle.run(prm, ref, E, i0, B, i0, work=wk)
    it = native.Integrator(dt, dx, 0.01, order=order, k_max=k_max, precision=native.PIC_FP64, qm=qm, capacity=n,
                           window=width, ring_levels=order + steps, field_time=field_time,
                           diagnostics=native.PIC_DIAG_WORK if work else 0)
    it.pic_particles_write(x, px, py, pz, status)
    for r in range(order + steps):
        it.pic_fields_upload(r - order, i0[r], E[r], B[r])
    st, _ = it.pic_push_step(0, steps, ok=OK)
    for name, g, o in zip(("x", "px", "py", "pz", "status"), it.read_numpy(),
                          (ref.x, ref.px, ref.py, ref.pz, ref.status)):
        np.testing.assert_array_equal(g, o, err_msg=name)
    for key in ("k_hist", "substeps", "n_star", "clamped", "out_of_window"):
        assert st.as_dict()[key] == ost.as_dict()[key], key
    if work:
        np.testing.assert_array_equal(it.work_read(), wk)
    it.close()


@pytest.mark.parametrize("n", [4095, 4096, 4097])
def test_as_many_electrons_as_nodes(n):
    _both(n, 4096, 3)


@pytest.mark.parametrize("order,qm,work,field_time", [(1, -1.0, False, 0), (2, -0.37, True, 1), (3, 1.0, True, 0),
                                                      (4, -1.0, False, 1), (5, -1.0, False, 0)])
def test_gathered_levels(order, qm, work, field_time):
    _both(2500, 1 << 15, order, qm=qm, work=work, field_time=field_time)


def test_a_large_window_does_not_slow_a_small_ensemble():
    """256 electrons, m = 1: a step in a window of 2^22 nodes costs what it costs in
    one of 2^12 (a pass over the nodes would take ten times as long)."""
    ms = {}
    for lw in (12, 22):
        width = 1 << lw
        it = native.Integrator(W.DT75, W.DT75 / 0.99, 1e30, precision=native.PIC_FP64, capacity=256, window=width,
                               ring_levels=12)
        z = torch.zeros(256, dtype=torch.float64, device="cuda")
        it.pic_particles_write(z + 3.0, z, z, z)
        f = torch.ones(width, dtype=torch.float64, device="cuda")
        for r in range(11):
            it.pic_fields_upload(r - 3, -8, f, f)
        t = []
        for _ in range(9):
            it.pic_particles_write(z + 3.0, z, z, z)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            it.pic_push_step(0, 8, want_stats=False)
            b.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(b))
        ms[lw] = sorted(t)[4]
        it.close()
    assert ms[22] < 3.0 * ms[12], ms


# one warp per electron up to four per SM, in one launch; the three passes beyond
@pytest.mark.parametrize("n", [1, 2, 33, 4 * 152, 4 * 152 + 1])
@pytest.mark.parametrize("order,work", [(1, False), (3, True), (5, False)])
def test_small_ensembles(n, order, work):
    _both(n, 64, order, k_max=5 if n < 100 else 3, work=work, qm=-1.0 if order < 5 else -0.37)


def test_small_ensembles_take_one_launch():
    it = native.Integrator(W.DT75, W.DT75 / 0.99, 0.01, precision=native.PIC_FP64, capacity=100, window=64,
                           ring_levels=8)
    z = np.zeros(100)
    it.pic_particles_write(z + 3.0, z, z, z)
    for r in range(7):
        it.pic_fields_upload(r - 3, -8, np.ones(64), np.ones(64))
    before = it.launches()
    it.pic_push_step(0, 4)
    assert it.launches() - before == 4
    it.close()
