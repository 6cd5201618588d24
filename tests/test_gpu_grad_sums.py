"""The gradient kernel's sums over a large batch, against the 64-bit sums of the
same operands: the network in FP64 with every operand rounded to BF16 where the
kernel rounds it.

Tolerance: a block adds m = 4 ceil(n / (64 * 152)) sums of 16 samples in FP32,
to nearest, so the rounding errors (half a unit of 2^-24 each, signs at random)
grow as sqrt(m); 4 sqrt(m) 2^-24 of the norm.  Sums that are truncated instead
are off by about m 2^-25, more than twice that at m = 432.
"""
from __future__ import annotations

import math

import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2102_10983_gb300 import native  # noqa: E402


def _bf(t):
    return t.float().bfloat16().double()


@pytest.mark.parametrize("n", [1 << 20, 4000001])
def test_sums_of_large_batches(n):
    gen = torch.Generator(device="cuda").manual_seed(n)
    X = torch.empty((n, 6), device="cuda").normal_(0, 2, generator=gen)
    # labels that follow the features: gradients that do not cancel over the batch
    Y = (X[:, 1].abs() * 1.5).clamp(0, 7).to(torch.uint8)
    P = omlp.init_params(3)
    net = native.Predictor()
    net.set_params(native.pack_params(P))
    g, _ = net.grad(X, Y)
    net.close()
    Q = {k: torch.as_tensor(v, device="cuda", dtype=torch.float64) for k, v in
         native.unpack_params(native.pack_params(P)).items()}
    x, W1, W2, W3 = _bf(X), _bf(Q["W1"]), _bf(Q["W2"]), _bf(Q["W3"])
    a1 = x @ W1.T + Q["b1"]
    h1 = _bf(a1.clamp(min=0))
    a2 = h1 @ W2.T + Q["b2"]
    h2 = _bf(a2.clamp(min=0))
    dz = torch.softmax(h2 @ W3.T + Q["b3"], 1)
    dz[torch.arange(n), Y.long()] -= 1
    dz = _bf(dz / n)
    da2 = _bf((dz @ W3) * (a2 > 0))
    da1 = _bf((da2 @ W2) * (a1 > 0))
    ref = torch.cat([v.reshape(-1) for v in (da1.T @ x, da1.sum(0), da2.T @ h1, da2.sum(0), dz.T @ h2, dz.sum(0))])
    ref = ref.cpu().numpy()
    m = 4 * math.ceil(n / (64 * 152))
    assert np.linalg.norm(g - ref) <= 4 * math.sqrt(m) * 2.0 ** -24 * np.linalg.norm(ref)
