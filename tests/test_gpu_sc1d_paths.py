"""The self-consistent loop where its fast paths end: electrons in no order
(every lane of a warp in a cell of its own) and many in one cell, charges
outside the integer conversions' range (negative, zero, above 2^52 units),
positions at both edges, |q/m| != 1.  Bit for bit against the oracle."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import pic1d
from paper_2102_10983_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2102_10983_gb300 import native  # noqa: E402


@pytest.mark.parametrize("n,cells,qm,order,spread", [
    (1, 16, -1.0, 1, "wide"), (33, 40, 0.6, 2, "wide"), (5000, 3000, -1.0, 3, "wide"),
    (5000, 300, -1.0, 5, "one cell"), (45000, 200, -2.0, 3, "wide")])
def test_sc1d_unsorted_electrons_and_odd_charges(n, cells, qm, order, spread):
    rng = np.random.Generator(np.random.PCG64(n + cells))
    dt = W.DT75
    dx = dt / 0.99
    s = rng.uniform(0.3, cells - 0.3, n) if spread == "wide" else 20.0 + rng.uniform(0.0, 1.0, n)
    x = s * dx
    px, py, pz = rng.normal(0.0, 1.5, (3, n))
    w = rng.uniform(0.001, 0.01, n)
    w[rng.random(n) < 0.1] *= -1.0
    w[rng.random(n) < 0.05] = 0.0
    w[rng.random(n) < 0.02] = 300.0  # above 2^52 units
    M = cells + 5
    k_max = 3
    amp = np.exp(rng.uniform(np.log(1e-3), np.log(20.0), M)) * rng.choice((-1.0, 1.0), M)
    lev = lambda: amp * rng.uniform(0.8, 1.2, M)  # noqa: E731
    E = [(lev(), lev()) for _ in range(order + 1)]
    B = [lev() for _ in range(order + 1)]
    prm = pic1d.Params(dt=dt, dx=dx, n_cells=cells, order=order, k_max=k_max, qm=qm)
    sim = pic1d.Pic1d(prm, x, px, py, pz, w, E, B)
    steps, worst = 3, 0.0
    for _ in range(steps):
        sim.step()
        worst = max(worst, sim.gauss()[0])
    g = native.Sc1d(dt, dx, cells, order=order, k_max=k_max, qm=qm, capacity=n, gauss_every=1)
    g.particles_write(x, px, py, pz, w)
    for l in range(order + 1):
        g.fields_write(l - order, E[l][0], E[l][1], B[l])
    st = g.step(0, steps)
    for name, a, b in zip(("x", "px", "py", "pz", "status"), g.read_numpy(),
                          (sim.x, sim.px, sim.py, sim.pz, sim.status)):
        np.testing.assert_array_equal(a, b, err_msg=name)
    for a, b in zip(g.fields_numpy(steps), (sim.E[-1][0], sim.E[-1][1], sim.B[-1])):
        np.testing.assert_array_equal(a, b)
    o = sim.stats
    assert list(st.k_hist) == list(o.k_hist)[:8]
    assert (st.substeps, st.n_star, st.clamped, st.frozen) == (o.substeps, o.n_star, o.clamped, o.frozen)
    assert st.gauss_residual == worst
    g.close()
