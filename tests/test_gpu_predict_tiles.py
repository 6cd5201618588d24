"""Inference at the edges of its tiles: a row's class does not depend on how many
rows there are, on the tile or the warpgroup that takes it, and nothing is
written past the last row.  Against the FP64 oracle where its top two logits
differ by more than 0.1 (BF16 operands, as in the other predictor tests)."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2102_10983_gb300 import native  # noqa: E402

MOST = 300_007


def _bf16(a):
    return torch.as_tensor(np.asarray(a, dtype=np.float32)).to(torch.bfloat16).to(torch.float64).numpy()


@pytest.mark.parametrize("n", [1, 31, 128, 129, 640, 19457, 97281, MOST])
def test_rows_are_independent(n):
    rng = np.random.default_rng(3)
    P = omlp.init_params(11)
    for k in P:
        if k.startswith("b"):
            P[k] = rng.normal(0, 0.3, P[k].shape)
    phi = np.arcsinh(rng.normal(0, 20, (MOST, 6))).astype(np.float32)
    net = native.Predictor()
    net.set_params(native.pack_params(P))
    X = torch.as_tensor(phi, device="cuda")
    pad = 192

    def infer(rows):
        out = torch.full((rows.shape[0] + pad,), 77, dtype=torch.uint8, device="cuda")
        net.infer(rows.contiguous(), out[:rows.shape[0]])
        torch.cuda.synchronize()
        assert (out[rows.shape[0]:] == 77).all()
        return out[:rows.shape[0]].cpu().numpy()

    whole = infer(X)
    np.testing.assert_array_equal(infer(X[:n]), whole[:n])
    np.testing.assert_array_equal(infer(X[:n].flip(0))[::-1], whole[:n])
    net.close()
    Pb = {k: (_bf16(v) if k.startswith("W") else np.asarray(v, np.float32).astype(np.float64))
          for k, v in P.items()}
    m = min(n, 20000)
    z, _ = omlp.forward(Pb, _bf16(phi[:m]))
    top = np.sort(z, 1)
    clear = top[:, -1] - top[:, -2] > 0.1 * np.maximum(1.0, np.abs(top[:, -1]))
    np.testing.assert_array_equal(whole[:m][clear], z.argmax(1)[clear])
