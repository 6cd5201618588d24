"""Loading and reading particles in the mixed layout against the definition in
numpy (x = (cell + frac) dx, frac FP32 in [0, 1); momenta rounded to FP32),
bit for bit: odd counts, arrays that start between 16-byte boundaries, values
at the ends of the integer conversions' range, ensembles of every size."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2102_10983_gb300 import native  # noqa: E402


def _inputs(n, seed, dx):
    """dx: one value per particle."""
    rng = np.random.Generator(np.random.PCG64(seed))
    s = rng.choice([rng.uniform(-5, 5, n), rng.uniform(0, 3e6, n), rng.uniform(-1e9, 1e9, n)], axis=0)
    s[rng.random(n) < 0.1] = np.round(s[rng.random(n) < 0.1][0] if n > 1 else 3.0)
    s[rng.random(n) < 0.1] = 1.0 - 2.0 ** -53
    s[rng.random(n) < 0.1] = 12345.0 - 2.0 ** -38  # frac rounds up to 1
    p = rng.normal(0, 1, (3, n)) * 10.0 ** rng.uniform(-50, 45, (3, n))
    p[rng.random((3, n)) < 0.1] = 0.0
    p[rng.random((3, n)) < 0.05] = -0.0
    # half-way between FP32 neighbours, the largest FP32 and what rounds past it
    p[rng.random((3, n)) < 0.1] = 1.0 + 2.0 ** -24
    p[rng.random((3, n)) < 0.1] = 1.0 + 3 * 2.0 ** -24
    p[rng.random((3, n)) < 0.05] = 3.4028235677973366e38
    return s * dx, p


def _expect(x, p, dx):
    s = x * (1.0 / dx)
    fl = np.floor(s)
    with np.errstate(over="ignore"):
        f = (s - fl).astype(np.float32)
        q = p.astype(np.float32).astype(np.float64)
    over = f >= 1
    f[over], fl[over] = 0.0, fl[over] + 1.0
    return (fl.astype(np.int32).astype(np.float64) + f.astype(np.float64)) * dx, q


def _device(a, shift):
    buf = torch.empty(a.shape[-1] + shift, dtype=torch.float64, device="cuda")[shift:]
    buf.copy_(torch.as_tensor(a))
    return buf


@pytest.mark.parametrize("n", [1, 2, 511, 100001])
@pytest.mark.parametrize("shift", [None, 0, 1])
def test_one_problem(n, shift):
    dx = 0.0846
    x, p = _inputs(n, n, np.full(n, dx))
    ex, ep = _expect(x, p, dx)
    it = native.Integrator(0.08, dx, 0.01, precision=native.PIC_MIXED, capacity=n)
    if shift is None:
        it.pic_particles_write(x, *p)
        got = it.read_numpy()[:4]
    else:
        it.pic_particles_write(_device(x, shift), *[_device(q, shift) for q in p])
        out = [torch.empty(n + shift, dtype=torch.float64, device="cuda")[shift:] for _ in range(4)]
        it.pic_particles_read(*out)
        torch.cuda.synchronize()
        got = [o.cpu().numpy() for o in out]
    it.close()
    for name, g, e in zip(("x", "px", "py", "pz"), got, (ex, *ep)):
        np.testing.assert_array_equal(g.view(np.int64), e.view(np.int64), err_msg=name)


@pytest.mark.parametrize("where", ["host", "device"])
def test_batch(where):
    sizes = [1, 0, 7, 1000, 0, 0, 3, 32769, 2, 0]
    dxs = [0.01 * (q + 1) / 0.99 for q in range(len(sizes))]
    n = sum(sizes)
    dx = np.repeat(dxs, sizes)
    x, p = _inputs(n, 9, dx)
    ex, ep = _expect(x, p, dx)
    b = native.Batch([dict(dt=0.5 * d, dx=d, psi_max=0.01, n_particles=c) for d, c in zip(dxs, sizes)])
    if where == "host":
        b.particles_write(x, *p)
    else:
        b.particles_write(_device(x, 0), *[_device(q, 0) for q in p])
    got = b.read_numpy()[:4]
    b.close()
    for name, g, e in zip(("x", "px", "py", "pz"), got, (ex, *ep)):
        np.testing.assert_array_equal(g.view(np.int64), e.view(np.int64), err_msg=name)
