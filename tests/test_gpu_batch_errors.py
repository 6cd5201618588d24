"""PIC_ETIMEOUT reporting of the batched ensembles, through the C ABI.

The batched stream waits, with a limit, for its staged tiles; a wait that gives
up sets the batch's device error word and leaves particles unpushed.  As in
test_gpu_errors.py the word is set from the host and the host's handling
checked: no device wait has to run out.
"""
from __future__ import annotations

import math

import numpy as np
import pytest

from paper_2102_10983_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2102_10983_gb300 import native  # noqa: E402


def _batch(levels=6):
    wl = W.Workload(name="berr", n_particles=400, a0=20.0, dt=W.DT75, dx=W.DT75 / 0.99, psi_max=0.01, order=3,
                    n_steps=0, x_lo=0.0, x_hi=2 * math.pi, window=256, lead=96)
    p = wl.order
    b = native.Batch([dict(dt=wl.dt, dx=wl.dx, psi_max=wl.psi_max, n_particles=wl.n_particles)] * 2, order=p,
                     window=wl.window, ring_levels=p + levels)
    ini = wl.particles()
    two = lambda v: np.ascontiguousarray(np.concatenate([v, v]))  # noqa: E731
    b.particles_write(two(ini.x), two(ini.px), two(ini.py), two(ini.pz))
    E, B, i0 = wl.levels(-p, p + levels)
    for r in range(p + levels):
        b.fields_upload(r - p, [i0[r]] * 2, np.stack([E[r]] * 2), np.stack([B[r]] * 2))
    return b


def test_push_step_reports_the_error_word_once():
    b = _batch()
    assert b.push_step(0, 1).error == 0
    b.inject_error(5)
    b.push_step(1, 1, want_stats=False)  # an asynchronous call keeps it
    st = native.PicStepStats()
    rc = native.lib().pic_batch_push_step(b.h, 2, 1, native.ctypes.byref(st))
    assert rc == native.PIC_ETIMEOUT and st.error == 5
    assert b"error word" in native.lib().pic_batch_last_error(b.h)
    assert b.push_step(3, 1).error == 0
    b.inject_error(1)
    with pytest.raises(native.PicError) as e:
        b.push_step(4, 1)
    assert e.value.code == native.PIC_ETIMEOUT
    b.close()


def test_autotune_reports_the_error_word_and_keeps_the_configuration():
    a, b = _batch(), _batch()
    b.inject_error(2)
    with pytest.raises(native.PicError) as e:
        b.autotune(0, 2)
    assert e.value.code == native.PIC_ETIMEOUT
    b.autotune(0, 2)  # reported once
    for u, v in zip(a.read_numpy(), b.read_numpy()):  # the particles are as they were
        assert np.array_equal(u, v)
    assert b.push_step(0, 2).error == 0
    a.close()
    b.close()
