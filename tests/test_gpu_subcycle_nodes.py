"""The mixed form's sub-cycles however an electron crosses its nodes: forward,
back and forth, several nodes or hardly any per macro step (cells from a
quarter to eight times c dt), out of the window's ends, k from 0 to 4.

One macro step from the same FP32-rounded state against the FP64 form.  Bound:
each of m sub-steps rounds the momentum, the rotation and the offset to a few
2^-24; an offset error of d cells moves the tent-interpolated field by at most
d times the node-to-node step.  So |dp| <= 64 (m + 16) 2^-24 (|p| + dt F)(1 +
Psi), F the largest field, Psi the step's rotation angle dt F / gamma; an
electron that took a wrong node would be off by about dt F / m.  Electrons
whose k differs (a criterion within FP32 rounding of a threshold) are left out;
there are few."""
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
@pytest.mark.parametrize("order", [1, 3, 5])
@pytest.mark.parametrize("schedule", [native.PIC_SCHED_PLAIN, native.PIC_SCHED_BINNED])
def test_any_crossing(ratio, order, schedule):
    n, width, dt = 20000, 64, W.DT75
    dx = dt / ratio
    rng = np.random.Generator(np.random.PCG64(int(100 * ratio) + order))
    top = 40.0
    shape = np.sin(np.arange(width) * rng.uniform(0.3, 1.0)) * top
    E, B = (np.array([shape * (1 + 0.1 * l) * s for l in range(order + 1)]) for s in (0.7, 1.0))
    x = rng.uniform(1.0, width - 1.0, n)
    edge = rng.random(n) < 0.1
    x[edge] = rng.choice((1.0, width - 2.0), edge.sum()) + rng.uniform(-0.6, 0.6, edge.sum())
    cell, frac = np.floor(x), (x - np.floor(x)).astype(np.float32)
    x = (cell + frac.astype(np.float64)) * dx
    p = (rng.normal(0, 1, (3, n)) * np.exp(rng.uniform(-2, 3, n))).astype(np.float32).astype(np.float64)
    E, B = E.astype(np.float32).astype(np.float64), B.astype(np.float32).astype(np.float64)
    out = []
    for precision, sched in ((native.PIC_FP64, 0), (native.PIC_MIXED, schedule)):
        it = native.Integrator(dt, dx, 0.01, order=order, precision=precision, schedule=sched, capacity=n,
                               window=width, ring_levels=order + 2, heavy_budget=100)
        it.pic_particles_write(x, *p)
        for l in range(order + 1):
            it.pic_fields_upload(l - order, 0, E[l], B[l])
        it.pic_push_step(0, 1, ok=(native.PIC_OK, native.PIC_ERANGE, native.PIC_EKMAX))
        out.append(it.read_numpy())
        it.close()
    (x0, *p0, s0), (x1, *p1, s1) = out
    same = s0 == s1
    assert same.mean() > 0.999 and (s0 >= native.PIC_STATUS_LOST).any()
    k = s0 & 7
    assert set(range(5)) <= set(k[same])
    F = 1.5 * top
    m = 4.0 ** k
    p_max = np.sqrt(np.sum(np.square(p0), axis=0)) + np.sqrt(np.sum(np.square(p), axis=0))
    gamma = np.sqrt(1 + np.minimum(np.sum(np.square(p0), axis=0), np.sum(np.square(p), axis=0)))
    tol = 64 * (m + 16) * 2.0 ** -24 * (p_max + dt * F) * (1 + dt * F / gamma)
    for a, b in zip(p0, p1):
        assert (np.abs(a - b)[same] <= tol[same]).all(), np.max((np.abs(a - b) / tol)[same])
