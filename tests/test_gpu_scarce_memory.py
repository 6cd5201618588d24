"""Contexts without room for their optional working memory: the node coefficient
tables of fewer steps, the queue of the sub-cycled electrons in slices, no node
fields.  They are created all the same and give the bits of the others.

The allocations are refused by a stand-in for cudaMalloc, loaded ahead of the
runtime in a child process, that returns cudaErrorMemoryAllocation for requests
of the sizes named in an environment variable and counts them.
"""
from __future__ import annotations

import ctypes
import hashlib
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2102_10983_gb300 import native
from paper_2102_10983_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
STAND_IN = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdlib.h>
#include <stddef.h>
int refused_allocations = 0;
int cudaMalloc(void** p, size_t n) {
  static int (*real)(void**, size_t) = 0;
  if (!real) {
    void* h = dlopen("libcudart.so.13", RTLD_NOW | RTLD_NOLOAD);
    if (!h) h = dlopen("libcudart.so.13", RTLD_NOW);
    if (!h) abort();
    real = (int (*)(void**, size_t))dlsym(h, "cudaMalloc");
  }
  const char* s = getenv("REFUSED_SIZES"); /* lo-hi[,lo-hi ...] */
  while (s && *s) {
    char* end;
    const size_t lo = strtoull(s, &end, 10), hi = strtoull(end + 1, &end, 10);
    if (n >= lo && n <= hi) {
      ++refused_allocations;
      *p = 0;
      return 2;
    }
    s = *end ? end + 1 : 0;
  }
  return real(p, n);
}
"""
N, ORDER, WIDTH = 300001, 3, 1 << 15


def _digest(arrays):
    return hashlib.sha256(b"".join(np.ascontiguousarray(a).tobytes() for a in arrays)).hexdigest()


def _electrons(n, width):
    rng = np.random.Generator(np.random.PCG64(n))
    x = np.sort(rng.uniform(2.0, width - 4.0, n)) * (W.DT75 / 0.99)
    return x, rng.normal(0, 2, n), rng.normal(0, 2, n), rng.normal(0, 1, n)


def _field(width, l):
    c = np.arange(width)
    return 30.0 * np.sin(0.02 * c + 0.1 * l), 30.0 * np.cos(0.017 * c + 0.1 * l)


def _push(precision, schedule, steps=6):
    it = native.Integrator(W.DT75, W.DT75 / 0.99, 0.01, order=ORDER, precision=precision, schedule=schedule, capacity=N,
                           window=WIDTH, ring_levels=ORDER + 1 + steps, heavy_budget=7, stream=0)
    it.pic_particles_write(*_electrons(N, WIDTH))
    for l in range(ORDER + steps):
        it.pic_fields_upload(l - ORDER, 0, *_field(WIDTH, l))
    st, _ = it.pic_push_step(0, steps, ok=(0, 4, 5))
    assert st.k_hist[0] > 0 and sum(st.k_hist[3:]) > 0
    out = it.read_numpy()
    it.close()
    return _digest(out + [np.array(list(st.k_hist))])


def _batch(steps=6):
    m, per, width = 60, 500, 1 << 14
    b = native.Batch([dict(dt=W.DT75, dx=W.DT75 / 0.99, psi_max=0.01, n_particles=per)] * m, order=ORDER, window=width,
                     ring_levels=ORDER + 1 + steps, stream=0)
    b.heavy_budget(7)
    b.particles_write(*[np.ascontiguousarray(np.tile(v, m)) for v in _electrons(per, width)])
    for l in range(ORDER + steps):
        b.fields_upload(l - ORDER, np.zeros(m), *[np.tile(f, (m, 1)) for f in _field(width, l)])
    st = b.push_step(0, steps)
    out = b.read_numpy()
    b.close()
    return _digest(out + [np.array(list(st.k_hist))])


def _sc1d(steps=2):
    cells = 4000
    g = native.Sc1d(W.DT75, W.DT75 / 0.99, cells, order=ORDER, capacity=N, gauss_every=1, stream=0)
    x, px, py, pz = _electrons(N, cells)
    g.particles_write(x, px, py, pz, np.full(N, 1e-3))
    for l in range(ORDER + 1):
        e, b = _field(cells + 5, l)
        g.fields_write(l - ORDER, 0.1 * e, e, b)
    st = g.step(0, steps)
    out = g.read_numpy() + g.fields_numpy(steps)
    g.close()
    return _digest(out + [np.array(list(st.k_hist))])


def _child():
    native.lib()
    out = [_push(native.PIC_FP64, native.PIC_SCHED_PLAIN), _push(native.PIC_MIXED, native.PIC_SCHED_BINNED), _batch(),
           _sc1d()]
    try:
        refused = ctypes.c_int.in_dll(ctypes.CDLL(None), "refused_allocations").value
    except ValueError:
        refused = 0
    print("RESULT", refused, *out)


def _sizes():
    """The requests to refuse: the queue of all electrons and of half of them (5
    bytes each, in 16s; FP64 form and coupled loop), 16, 8 and 4 tables, the batch's 8
    and 4, the node fields of the FP64 form and of the loop."""
    table, btable = WIDTH * 8 * (ORDER + 1), 60 * (1 << 14) * 8 * (ORDER + 1)
    all_of_them = (N + 15) // 16 * 16
    half = (all_of_them // 2 + 15) // 16 * 16
    return [5 * all_of_them, 5 * half, 16 * table, 8 * table, 4 * table, 8 * btable, 4 * btable, 32 * WIDTH, 48 * 4005]


def test_scarce_memory_changes_nothing(tmp_path):
    native.lib()  # built before the children need it
    src, so = tmp_path / "stand_in.c", tmp_path / "stand_in.so"
    src.write_text(STAND_IN)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(so), str(src), "-ldl"], check=True)
    got = []
    for env in ({}, {"LD_PRELOAD": str(so), "REFUSED_SIZES": ",".join(f"{v}-{v}" for v in _sizes())}):
        r = subprocess.run([sys.executable, os.path.abspath(__file__)], env={**os.environ, "PYTHONPATH": ROOT, **env},
                           capture_output=True, text=True, timeout=300)
        line = [v for v in r.stdout.splitlines() if v.startswith("RESULT")]
        assert r.returncode == 0 and line, r.stderr[-2000:]
        got.append(line[0].split()[1:])
    assert int(got[0][0]) == 0 and int(got[1][0]) == 11  # FP64 2 + 1, tables 3 and 2, loop 2 + 1
    assert got[0][1:] == got[1][1:]


if __name__ == "__main__":
    _child()
