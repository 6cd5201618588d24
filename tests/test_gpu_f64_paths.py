"""The FP64 push where its fast paths end: node coordinates outside [1, 2^21)
(read off the significand inside, by floor outside), operands outside the
domain of the integer division and square root, |q/m| != 1, large k_prev, and
every number of electrons per warp of the sub-cycle kernel.  Bit for bit
against the oracle (no tolerance)."""
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


def _both(n, origin, qm, order, k_max, extreme, seed, work=False, dt=W.DT75, steps=2):
    rng = np.random.Generator(np.random.PCG64(seed))
    dx = dt / 0.99
    width = 64
    i0 = np.full(order + steps, origin, dtype=np.int64)
    # per-node amplitudes over the criterion's whole range, levels varying around them
    amp = np.exp(rng.uniform(np.log(1e-3), np.log(300.0), width)) * rng.choice((-1.0, 0.0, 1.0), width, p=(.45, .1, .45))
    E, B = (amp * rng.uniform(0.5, 1.5, (order + steps, width)) for _ in range(2))
    x = (origin + rng.uniform(-0.5, width + 0.5, n)) * dx  # some outside the window
    px, py, pz = rng.normal(0.0, 2.0, (3, n))
    rest = rng.random(n) < 0.2
    px[rest] = py[rest] = pz[rest] = 0.0
    if extreme:
        E[:, ::7], B[:, ::5], B[:, 3::11] = 1e-310, 0.0, 1e-200
        B[:, 4::13] = 1e150
        px[::9], py[::14], pz[::17] = 1e160, 1e-320, 1e100
    status = rng.integers(0, 13, n).astype(np.uint8)
    status[rng.random(n) < 0.02] |= native.PIC_STATUS_LOST
    prm = oracle.Params(dt=dt, dx=dx, psi_max=0.01, order=order, k_max=k_max, qm=qm)
    ref = oracle.Particles(x, px, py, pz, status)
    wk = np.zeros(n) if work else None
    ost = oracle.run(prm, ref, E, i0, B, i0, work=wk)
    it = native.Integrator(dt, dx, 0.01, order=order, k_max=k_max, precision=native.PIC_FP64, qm=qm,
                           capacity=n, window=width, ring_levels=order + steps,
                           diagnostics=native.PIC_DIAG_WORK if work else 0)
    it.pic_particles_write(x, px, py, pz, status)
    for r in range(order + steps):
        it.pic_fields_upload(r - order, i0[r], E[r], B[r])
    st, _ = it.pic_push_step(0, steps, ok=OK)
    got = it.read_numpy()
    for name, g, o in zip(("x", "px", "py", "pz", "status"), got,
                          (ref.x, ref.px, ref.py, ref.pz, ref.status)):
        np.testing.assert_array_equal(g, o, err_msg=name)
    for key in ("k_hist", "substeps", "n_star", "clamped", "out_of_window"):
        assert st.as_dict()[key] == ost.as_dict()[key], key
    if work:
        np.testing.assert_array_equal(it.work_read(), wk)
    it.close()
    return st


@pytest.mark.parametrize("origin", [-40, -2, 0, (1 << 21) - 30, 1 << 30])
@pytest.mark.parametrize("qm", [-1.0, 1.0, -0.37])
def test_node_coordinates_and_charge(origin, qm):
    _both(700, origin, qm, 3, 3, False, seed=abs(origin) % 1000 + int(100 + 10 * qm))


@pytest.mark.parametrize("order,work", [(1, False), (3, True), (5, False)])
def test_operands_outside_the_integer_domain(order, work):
    _both(900, 100, -1.0, order, 2, True, seed=order, work=work)


# one electron; a few of each k (one per warp); then so many that warps hold 2 .. 32
@pytest.mark.parametrize("n,k_max", [(1, 7), (31, 6), (2000, 5), (9000, 3), (60000, 1)])
def test_electrons_per_warp(n, k_max):
    st = _both(n, 0, -1.0, 3, k_max, False, seed=n)
    if n >= 2000:
        assert min(st.k_hist[:k_max + 1]) > 0  # every k occurs


def test_tiny_step_and_threshold():
    """A macro step whose powers of four leave the normal range, and a criterion
    scale outside the FP32 test's."""
    _both(300, 10, -1.0, 2, 2, False, seed=5, dt=1e-290)
