"""The study kernel at every order, both field-time readings, a charge other
than one, k above 2 (weights formed 32 sub-steps at a time) and cells of very
different size (one node, several nodes or none crossed in a macro step),
through a short pulse, against the study oracle: k of every step exactly, the
errors within four times the spread of the oracle's own runs with every field
sample moved by 1 and 4 ulps (as tests/test_gpu_study.py)."""
from __future__ import annotations

import ctypes

import pytest

from oracle import study
from paper_2102_10983_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2102_10983_gb300 import native  # noqa: E402

ULP = 2.0 ** -52
SHAPES = [(1, 0, -1.0, 0.99), (2, 1, -1.0, 3.1), (3, 0, -0.5, 0.99), (3, 1, -1.0, 0.2), (4, 0, -1.0, 0.99),
          (5, 1, 0.7, 2.3), (5, 0, -1.0, 0.99)]


def _oracle(order, field_time, qm, ratio, steps, scale):
    return study.TrjParams(6.0, 18.0, 6.0, W.DT75, W.DT75 / ratio, 0.004, qm, order, 7, field_time, 0, steps, 0.0,
                           scale)


@pytest.mark.parametrize("order,field_time,qm,ratio", SHAPES)
def test_study_shapes(order, field_time, qm, ratio):
    steps = 220
    q = native.PicStudyCase(6.0, 18.0, 6.0, W.DT75, W.DT75 / ratio, 0.004, qm, order, 7, field_time, 1, steps)
    g = native.PicStudyResult()
    assert native.lib().pic_study_run(ctypes.byref(q), 1, ctypes.byref(g), None) == native.PIC_OK
    got = g.as_dict()
    r, *moved = study.run([_oracle(order, field_time, qm, ratio, steps, f)
                           for f in (1.0, 1 + ULP, 1 - ULP, 1 + 4 * ULP, 1 - 4 * ULP)])
    assert got["k_hist"] == r["k_hist"] and sum(got["k_hist"][3:]) > 0
    for key in ("eps_dephasing", "eps_energy", "gamma_max"):
        spread = max(abs(m[key] - r[key]) for m in moved)
        assert abs(got[key] - r[key]) <= 4.0 * spread + 1e-13 * abs(r[key]), (key, got[key], r[key], spread)
