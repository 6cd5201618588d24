"""Studies of many electrons (one thread each) beside the same cases one at a time
(one warp per electron): every order, both field-time readings, |q/m| != 1, k
above 2 and cells of very different size.  The two forms take the same
operations, so every result is equal; and many electrons share the FP64 unit."""
from __future__ import annotations

import time

import pytest

from paper_2102_10983_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2102_10983_gb300 import native  # noqa: E402
from test_gpu_study_paths import SHAPES  # noqa: E402


def _run(cases):
    arr, out = (native.PicStudyCase * len(cases))(*cases), (native.PicStudyResult * len(cases))()
    assert native.lib().pic_study_run(arr, len(cases), out, None) == native.PIC_OK
    return [r.as_dict() for r in out]


def test_many_electrons_take_the_same_steps():
    shapes = SHAPES + [(2, 0, -1.0, 0.99), (4, 1, -2.0, 1.7)]
    sizes = [256, 255, 33, 32, 31, 1]
    cases = [native.PicStudyCase(6.0 + 0.01 * q, 18.0, 6.0, W.DT75, W.DT75 / r, 0.004, qm, o, 7, ft,
                                 sizes[q % len(sizes)] if q < 18 else 256, 220)
             for q, (o, ft, qm, r) in enumerate(shapes * 5)]
    assert sum(c.n_electrons for c in cases) > 32 * 152
    alone = [_run([c])[0] for c in cases]
    assert any(sum(r["k_hist"][3:]) > 0 for r in alone)
    assert _run(cases) == alone


def test_many_electrons_cost_less_than_one_each():
    """81,920 electrons take at most 60 times as long as one: a warp each, they
    would take 90 times as long."""
    def seconds(n_cases, n_e):
        cases = [dict(a0=5.0, order=3, psi_max=0.01, res=75, n_electrons=n_e, n_steps=1500)] * n_cases
        t = []
        for _ in range(3):
            t0 = time.perf_counter()
            native.study_run(cases)
            t.append(time.perf_counter() - t0)
        return min(t)
    assert seconds(320, 256) < 60 * seconds(1, 1)
