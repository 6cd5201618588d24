"""What this library is timed on: the passes its users make through its public
entry points (paper_2102_10983_gb300.native, the binding of include/*.h).

A pass of a push is a whole use of the integrator: load the electrons, store
the field levels, take the macro steps, read the electrons and the counters.
So it does the same work each time it is called on a state.  Inputs are drawn
on the GPU from the seed: electrons as they are behind the switched-on wave's
front (phase xi from the exact orbit of an electron with gamma - p_x = R, R
spread as that front spreads it), and the plane wave's levels.

exact() is the method of the paper in plain FP64 torch on the same inputs.
"""
from __future__ import annotations

import ctypes
import dataclasses
import math

import numpy as np
import torch

from paper_2102_10983_gb300 import native
from paper_2102_10983_gb300 import workloads as W

DEV = "cuda"
TWO_PI = 2.0 * math.pi


def listed():
    base = {"order": 3, "field_time": 0, "a0": 150.0, "thermal": True, "res": 75, "psi": 0.01,
            "work": False}
    push = dict(base, kind="push", carry=0, every=0)
    return [
        # the test-particle configuration: 256 electrons, the default form (FP64), one step
        # per call after that step's level arrives from the host: launches and latency
        dict(push, name="f64_256_by_step", form="f64", n=256, a0=100.0, thermal=False, start=60,
             steps=16, window=256, lead=96, span=1.0, calls="each", levels="host"),
        # the same loop in the mixed form with the binned schedule (a solver's small test run)
        dict(push, name="mixed_300_by_step", form="binned", n=300, a0=100.0, thermal=False, start=60,
             steps=16, window=256, lead=96, span=1.0, calls="each", levels="host"),
        # the FP64 form on a Maxwellian ensemble in the a0 = 150 wave: the reference run that
        # the mixed form is validated against
        dict(push, name="f64_1M", form="f64", n=1 << 20, start=2400, steps=2, window=32768,
             lead=0, span=64.0, calls="one", levels="device"),
        # the headline ensemble: 16.8M electrons, mixed form, binned schedule, steps in one call
        dict(push, name="mixed_16M", form="binned", n=1 << 24, start=2400, steps=8, window=32768,
             lead=0, span=64.0, calls="one", levels="device"),
        # a ragged ensemble at fifth order with the other field-time reading
        dict(push, name="mixed_1000003_order5", form="binned", n=1000003, order=5, field_time=1,
             start=1200, steps=8, window=32768, lead=0, span=64.0, calls="one",
             levels="device"),
        # the coupled loop: a field solver uploads one level per step from pinned host memory,
        # learned binning, long sub-cycles carried from call to call, counters read every step
        dict(push, name="predicted_4M_by_step", form="predicted", n=1 << 22, start=2400, steps=8,
             window=32768, lead=0, span=64.0, calls="each", levels="pinned", carry=1, every=64),
        # a host program that owns all device memory: its own arrays, nothing allocated
        dict(base, name="noalloc_65536", kind="noalloc", n=65536, start=600, steps=4, window=1024,
             lead=200, span=4.0),
        # the learned predictor on its own: every electron's class for the next step
        dict(push, name="predict_8M", kind="predict", form="binned", n=1 << 23, start=2400, steps=1,
             window=32768, lead=0, span=64.0, via="fused"),
        # its training loop: Adam on mini-batches of logged pairs
        {"name": "train_8192", "kind": "train", "batch": 8192, "iters": 8, "lr": 2e-3},
        # a parameter scan: 512 ensembles cycling a0 x resolution x Psi_max, log-uniform sizes
        {"name": "batch_512", "kind": "batch", "ens": 512, "smallest": 1000, "largest": 100000,
         "order": 3, "start": 600, "steps": 8, "window": 2048, "graph": True},
        # the self-consistent laser-plasma loop: 100 electrons per cell, Gauss's law checked
        {"name": "sc1d_20000", "kind": "sc1d", "cells": 20000, "ppc": 100, "a0": 150.0, "order": 3,
         "field_time": 0, "psi": 0.01, "start": 2400, "steps": 4, "gauss": 1},
        # single-electron studies: interpolation orders 1, 3 and 5, 64 electrons each, up to the
        # middle of the pulse
        {"name": "study_a0_5", "kind": "study", "a0": 5.0, "orders": "135", "res": 75, "psi": 0.01,
         "electrons": 64, "steps": 2000},
    ]


def draw(rng):
    """One more case of the same ranges."""
    def logn(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return min(max(n | 1 if rng.random() < 0.5 else n, lo), hi)

    base = {"order": rng.choice((1, 2, 3, 3, 3, 4, 5)), "field_time": rng.choice((0, 0, 0, 1)),
            "a0": rng.choice((10.0, 30.0, 100.0, 150.0, 300.0)), "thermal": rng.random() < 0.7,
            "res": rng.choice((50, 75, 75, 150)), "psi": rng.choice((0.003, 0.01, 0.01, 0.03)),
            "work": False}
    grid = {"start": rng.randint(300, 2400), "window": 32768, "lead": 0, "span": 64.0,
            "carry": 0, "every": 0}
    near = {"start": rng.randint(300, 700), "window": 1024, "lead": 300, "span": 1.0}
    kind = rng.choice(("f64", "f64", "binned", "binned", "binned", "predicted", "noalloc", "predict",
                       "train", "batch", "sc1d", "study"))
    calls = {"calls": rng.choice(("one", "each")), "levels": rng.choice(("host", "pinned", "device"))}
    if kind == "f64":
        n = logn(200, 1 << 20)
        c = dict(base, kind="push", form="f64", n=n, steps=rng.randint(1, 2 if n > 1 << 16 else 12),
                 **grid, **calls)
        return dict(c, work=rng.random() < 0.3)
    if kind == "binned":
        n = logn(200, 1 << 23)
        small = dict(carry=0, every=0, **near) if n < 20000 else grid
        c = dict(base, kind="push", form="binned", n=n, steps=rng.randint(2, 12), **small, **calls)
        return dict(c, carry=1 if c["calls"] == "each" and rng.random() < 0.4 else 0)
    if kind == "predicted":
        return dict(base, kind="push", form="predicted", n=logn(20000, 1 << 22), steps=rng.randint(2, 10),
                    **dict(grid, carry=rng.choice((0, 1)), every=rng.choice((1, 5, 64))), **calls)
    if kind == "noalloc":
        return dict(base, kind="noalloc", n=logn(200, 65536), steps=rng.randint(1, 8), **near)
    if kind == "predict":
        return dict(base, kind="predict", form="binned", n=logn(1000, 1 << 23), steps=1,
                    via=rng.choice(("fused", "features")), **grid)
    if kind == "train":
        return {"kind": "train", "batch": logn(256, 16384), "iters": rng.randint(2, 10), "lr": 2e-3}
    if kind == "batch":
        return {"kind": "batch", "ens": logn(2, 512), "smallest": 500, "largest": logn(2000, 90000),
                "order": base["order"], "start": rng.randint(300, 1500), "steps": rng.randint(2, 10),
                "window": 2048, "graph": rng.random() < 0.5}
    if kind == "sc1d":
        return {"kind": "sc1d", "cells": logn(6000, 20000), "ppc": rng.randint(4, 90), "a0": base["a0"],
                "order": base["order"], "field_time": base["field_time"], "psi": base["psi"],
                "start": rng.randint(600, 2400), "steps": rng.randint(1, 4), "gauss": rng.choice((0, 1))}
    return {"kind": "study", "a0": rng.choice((2.0, 5.0, 10.0)), "orders": rng.choice(("1", "13", "3", "135", "24")),
            "res": rng.choice((50, 75, 75)), "psi": rng.choice((0.01, 0.03)),
            "electrons": rng.randint(1, 64), "steps": rng.choice((600, 1500, 2000))}


def _rng(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) % (1 << 62))


def _f64(*shape):
    return torch.empty(shape, dtype=torch.float64, device=DEV)


# ---------------------------------------------------------------- inputs

def _electrons(g, n, a0, t0, span, thermal, xi_cap):
    """n electrons of the switched-on wave at time t0, in order of where they started
    (uniform in [0, span lambda)); a0, t0, xi_cap: numbers or one value per electron."""
    u = _f64(n).uniform_(generator=g)
    z = _f64(4, n).normal_(generator=g)
    x0 = torch.sort(u).values * (span * TWO_PI)
    as_t = lambda v: v if torch.is_tensor(v) else torch.full((), float(v), dtype=torch.float64, device=DEV)  # noqa: E731
    a0, t0, cap = as_t(a0), as_t(t0), as_t(xi_cap)
    f = torch.clamp(a0 / 150.0, max=1.0)
    R = torch.exp(torch.log1p(2.4 * f) + 0.7 * f * z[0])
    R = torch.minimum(torch.clamp(R, min=0.45), 1.0 + 24.0 * f)
    tau = torch.clamp(t0 - x0, min=0.0)
    p, q = (1.0 + R * R) / (2.0 * R * R), a0 * a0 / (2.0 * R * R)
    lo, hi = torch.zeros_like(x0), torch.minimum(tau / p, cap)
    for _ in range(45):  # tau = p xi + q (xi / 2 - sin(2 xi) / 4) increases with xi
        mid = 0.5 * (lo + hi)
        late = p * mid + q * (0.5 * mid - 0.25 * torch.sin(2.0 * mid)) > tau
        hi = torch.where(late, mid, hi)
        lo = torch.where(late, lo, mid)
    xi = 0.5 * (lo + hi)
    hit = tau > 0.0
    th = W.MAXWELL_10KEV_SIGMA if thermal else 0.0
    py = torch.where(hit, a0 * torch.sin(xi), torch.zeros_like(xi)) + th * z[1]
    pz = th * z[2]
    px = torch.where(hit, (1.0 + py * py + pz * pz - R * R) / (2.0 * R), th * z[3])
    x = torch.where(hit, t0 - xi, x0)
    return [v.contiguous() for v in (x, px, py, pz)]


def _level(a0, dt, dx, n, i0, width):
    """Level n (E_y at n dt, B_z at (n + 1/2) dt) of the switched-on wave on `width` nodes from i0;
    numbers, or columns of one value per ensemble."""
    c = torch.arange(width, dtype=torch.float64, device=DEV)
    xe = n * dt - (i0 + c) * dx
    xb = (n + 0.5) * dt - (i0 + c + 0.5) * dx
    return tuple(torch.where(x > 0, -a0 * torch.cos(x), torch.zeros_like(x)).contiguous() for x in (xe, xb))


def _push_inputs(c, seed):
    dt = TWO_PI / c["res"]
    dx = dt / 0.99
    t0 = c["start"] * dt
    # a fixed window as of the full-size ensembles, or one that follows the front
    first, count = c["start"] - c["order"], c["order"] + c["steps"]
    if c["lead"]:
        i0 = W.chase_origins(first, count, dt, dx, c["window"], c["lead"])
        cap = max(1.0, t0 - (float(i0[-1]) + 3 + count) * dx)
    else:
        i0 = np.full(count, -512, dtype=np.int64)
        cap = t0 + 500 * dx
    parts = _electrons(_rng(seed), c["n"], c["a0"], t0, c["span"], c["thermal"], cap)
    levels = [_level(c["a0"], dt, dx, float(first + r), float(i0[r]), c["window"]) for r in range(count)]
    return dt, dx, i0, parts, levels


def _batch_inputs(c, seed):
    """Ensembles cycling a0 x lambda/(c dt) x Psi_max, electrons starting within a wavelength."""
    m, p = c["ens"], c["order"]
    r = np.random.Generator(np.random.PCG64(m))  # the sizes are the scan's, not the seed's
    sizes = np.round(np.exp(r.uniform(math.log(c["smallest"]), math.log(c["largest"]), m))).astype(np.int64)
    a0 = np.array([(10.0, 30.0, 100.0, 300.0)[q % 4] for q in range(m)])
    dt = np.array([TWO_PI / (25, 50, 75, 150)[(q // 4) % 4] for q in range(m)])
    dx = dt / 0.99
    psi = [(0.003, 0.01, 0.03)[(q // 16) % 3] for q in range(m)]
    ens = [dict(dt=dt[q], dx=dx[q], psi_max=psi[q], n_particles=int(sizes[q])) for q in range(m)]
    count = p + c["steps"]
    lev = (c["start"] - p + np.arange(count))[:, None]
    i0 = (np.floor(lev * dt / dx) + np.ceil(TWO_PI / dx) + 16 - c["window"]).astype(np.int64)
    col = lambda v: torch.as_tensor(v, dtype=torch.float64, device=DEV)  # noqa: E731
    eid = torch.repeat_interleave(torch.arange(m, device=DEV), torch.as_tensor(sizes, device=DEV))
    t0 = c["start"] * dt
    cap = t0 - (i0[-1] + 3) * dx
    x, px, py, pz = _electrons(_rng(seed), int(sizes.sum()), col(a0)[eid], col(t0)[eid], 1.0, False, col(cap)[eid])
    levels = [_level(col(a0)[:, None], col(dt)[:, None], col(dx)[:, None], float(lev[r, 0]),
                     col(i0[r])[:, None], c["window"]) for r in range(count)]
    return ens, eid, i0, [x, px, py, pz], levels


def _sc1d_inputs(c, seed):
    """The laser-plasma configuration after `start` steps: electrons on their vacuum orbits
    (R = 1) in the pulse, a little thermal scatter from the seed."""
    wl = dataclasses.replace(W.laser_plasma_c5(c["cells"], c["ppc"], c["a0"]), order=c["order"], psi_max=c["psi"])
    # the published grid is 20,000 cells: a shorter one starts its plasma within the grid
    top = min(wl.x_top, 0.6 * c["cells"] * wl.dx)
    front = wl.x_front + (top - wl.x_top)
    t0 = c["start"] * wl.dt
    wl = dataclasses.replace(wl, x_top=top, x_front=front + t0)
    x0, _, _, _, w = wl.particles()
    xi = np.linspace(0.0, wl.duration, 40001)
    a = wl.a(xi)
    F = xi + np.concatenate(([0.0], np.cumsum(0.25 * (a[1:] ** 2 + a[:-1] ** 2) * np.diff(xi))))
    ph = np.where(x0 - front < t0, np.interp(t0 - (x0 - front), F, xi), -1.0)
    hit = ph > 0.0
    x = np.where(hit, front + t0 - ph, x0)
    keep = x < (c["cells"] - 8) * wl.dx
    x, w, ph, hit = x[keep], w[keep], ph[keep], hit[keep]
    r = np.random.Generator(np.random.PCG64(seed))
    py = np.where(hit, wl.a(np.where(hit, ph, 0.0)), 0.0) + 1e-3 * r.standard_normal(x.size)
    px = 0.5 * py * py
    to = lambda v: torch.as_tensor(np.ascontiguousarray(v), device=DEV)  # noqa: E731
    E, B = wl.field_history()
    levels = [[to(v) for v in (E[l][0], E[l][1], B[l])] for l in range(c["order"] + 1)]
    return wl, [to(v) for v in (x, px, py, np.zeros_like(x), w)], levels


def _net_params(seed):
    """A predictor as training leaves it: logits linear in z = asinh|B| - log gamma, class k
    from z's distance to the criterion's thresholds; scattered small weights beside that."""
    r = np.random.Generator(np.random.PCG64(seed))
    P = {k: r.normal(0.0, 0.004, s) for k, s in (("W1", (64, 6)), ("b1", (64,)), ("W2", (64, 64)), ("b2", (64,)),
                                                 ("W3", (8, 64)), ("b3", (8,)))}
    P["W1"][0, 1], P["W1"][0, 5], P["b1"][0] = 1.0, -1.0, 12.0
    P["W2"][0, 0] = 1.0
    first = math.log(2.0) + math.log(2.0 * 0.01 / W.DT75)  # k = 0 below this z
    for k in range(8):
        P["W3"][k, 0] = float(k)
        P["b3"][k] = -k * (first + 12.0) - 0.5 * k * (k - 1) * math.log(4.0)
    return native.pack_params(P)


def _train_inputs(c, seed):
    """Logged pairs as the test-particle run gives them: features of electrons in the wave, the
    criterion's k; and He-uniform starting weights."""
    n = c["batch"] * c["iters"]
    g = _rng(seed)
    x, px, py, pz = _electrons(g, n, 100.0, 200 * W.DT75, 2.0, False, 20.0)
    xi = 200 * W.DT75 - x
    b = torch.where(xi > 0, 100.0 * torch.cos(xi).abs(), torch.zeros_like(xi))
    gamma = torch.sqrt(1.0 + px * px + py * py + pz * pz)
    k = torch.ceil(torch.log2(torch.clamp(b * W.DT75 / (2.0 * gamma) / 0.01, min=1e-9)) / 2.0).clamp(0, 7)
    phi = torch.stack([torch.asinh(b), torch.asinh(b), torch.asinh(px), torch.asinh(py), torch.asinh(pz),
                       torch.log(gamma)], dim=1)
    perm = torch.randperm(n, device=DEV, generator=g)
    r = np.random.Generator(np.random.PCG64(seed))
    P = {"b1": np.zeros(64), "b2": np.zeros(64), "b3": np.zeros(8)}
    for name, (o, i) in (("W1", (64, 6)), ("W2", (64, 64)), ("W3", (8, 64))):
        P[name] = r.uniform(-1, 1, (o, i)) * math.sqrt(6.0 / i)
    return phi[perm].float().contiguous(), k[perm].to(torch.uint8).contiguous(), native.pack_params(P)


def _study_cases(c):
    dt = TWO_PI / c["res"]
    steps = c["steps"] or W.study_steps(c["a0"], dt, x_span=TWO_PI * (c["electrons"] - 1) / c["electrons"])
    return [dict(a0=c["a0"], order=int(o), psi_max=c["psi"], res=c["res"], n_electrons=c["electrons"],
                 n_steps=steps) for o in c["orders"]]


# ---------------------------------------------------------------- states

def prepare(c, seed):
    kind, s = c["kind"], {"case": c}
    if kind in ("push", "predict"):
        dt, dx, i0, parts, levels = _push_inputs(c, seed)
        form = c["form"]
        s["parts"], s["i0"], s["first"] = parts, [int(v) for v in i0], c["start"] - c["order"]
        s["out"] = [torch.empty_like(v) for v in parts] + [torch.empty(c["n"], dtype=torch.uint8, device=DEV)]
        s["integ"] = native.Integrator(
            dt, dx, c["psi"], order=c["order"], precision=native.PIC_FP64 if form == "f64" else native.PIC_MIXED,
            field_time=c["field_time"], capacity=c["n"], window=c["window"],
            ring_levels=c["order"] + 2 + c["steps"], carry=c["carry"],
            schedule={"f64": native.PIC_SCHED_PLAIN, "binned": native.PIC_SCHED_BINNED,
                      "predicted": native.PIC_SCHED_PREDICTED}[form],
            diagnostics=native.PIC_DIAG_WORK if c["work"] else 0)
        if c["work"]:
            s["done"] = torch.empty_like(parts[0])
        if form == "predicted" or kind == "predict":
            s["net"] = native.Predictor(seed=int(seed))
            s["net"].set_params(_net_params(seed))
            if form == "predicted":
                s["integ"].attach_predictor(s["net"], c["every"])
        if kind == "predict":
            s["phi"] = torch.empty((c["n"], 6), dtype=torch.float32, device=DEV)
            s["pred"] = torch.empty(c["n"], dtype=torch.uint8, device=DEV)
            s["levels"] = levels
            # the electrons are in the integrator already, as after its last step
            s["integ"].pic_particles_write(*parts)
            for r, (E, B) in enumerate(levels):
                s["integ"].pic_fields_upload(s["first"] + r, s["i0"][r], E, B)
        elif c["levels"] == "device":
            s["levels"] = levels
        else:
            host = [[v.cpu() for v in lv] for lv in levels]
            s["levels"] = [[v.pin_memory() for v in lv] if c["levels"] == "pinned" else
                           [v.numpy() for v in lv] for lv in host]
    elif kind == "noalloc":
        dt, dx, i0, parts, levels = _push_inputs(c, seed)
        sx = parts[0] * (1.0 / dx)
        frac = (sx - sx.floor()).float()
        over = frac >= 1.0
        s["cell"] = (sx.floor() + over).to(torch.int32)
        s["from"] = [s["cell"], torch.where(over, torch.zeros_like(frac), frac)] + [v.float() for v in parts[1:]]
        s["from"].append(torch.zeros(c["n"], dtype=torch.uint8, device=DEV))
        s["out"] = [torch.empty_like(v) for v in s["from"]]
        nodes = torch.arange(c["window"], device=DEV)
        s["levels"] = [[torch.empty(c["window"], device=DEV).index_copy_(0, (nodes + int(i0[r])) & (c["window"] - 1),
                                                                        v.float()) for v in lv]
                       for r, lv in enumerate(levels)]
        s["i0"] = np.ascontiguousarray(i0)
        s["prm"] = native.PicParams(dt, dx, c["psi"], -1.0, c["order"], 7, native.PIC_MIXED, c["field_time"],
                                    native.PIC_SCHED_BINNED)
        s["E"], s["B"] = ((ctypes.c_void_p * len(levels))(*[lv[k].data_ptr() for lv in s["levels"]]) for k in (0, 1))
    elif kind == "train":
        s["X"], s["Y"], s["params"] = _train_inputs(c, seed)
        s["net"] = native.Predictor(seed=int(seed))
    elif kind == "batch":
        ens, _, i0, s["parts"], s["levels"] = _batch_inputs(c, seed)
        s["i0"] = i0
        s["stream"] = torch.cuda.Stream()  # graph capture wants a stream of its own
        s["batch"] = native.Batch(ens, order=c["order"], window=c["window"],
                                  ring_levels=c["order"] + 2 + c["steps"], stream=s["stream"])
        s["batch"].config(chunk=512, blocks_per_sm=4, use_graph=c["graph"])
        s["out"] = [torch.empty_like(v) for v in s["parts"]]
        s["out"].append(torch.empty(s["parts"][0].numel(), dtype=torch.uint8, device=DEV))
    elif kind == "sc1d":
        wl, s["parts"], s["levels"] = _sc1d_inputs(c, seed)
        n = s["parts"][0].numel()
        s["loop"] = native.Sc1d(wl.dt, wl.dx, c["cells"], psi_max=c["psi"], order=c["order"],
                                field_time=c["field_time"], capacity=n, gauss_every=c["gauss"])
        s["out"] = [torch.empty_like(v) for v in s["parts"][:4]] + [torch.empty(n, dtype=torch.uint8, device=DEV)]
        s["fields"] = [_f64(c["cells"] + 5) for _ in range(3)]
    else:
        # a study takes parameters only: the seed moves a0 a little
        r = np.random.Generator(np.random.PCG64(seed))
        s["cases"] = [dict(q, a0=q["a0"] * (1.0 + 1e-3 * r.random())) for q in _study_cases(c)]
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------- passes

def _counts(st):
    return np.array(list(st.k_hist) + [st.substeps, st.n_star, st.clamped], dtype=np.int64)


OK = (native.PIC_OK, native.PIC_ERANGE, native.PIC_EKMAX)


def run(s):
    return {"push": _run_push, "noalloc": _run_noalloc, "predict": _run_predict, "train": _run_train,
            "batch": _run_batch, "sc1d": _run_sc1d, "study": _run_study}[s["case"]["kind"]](s)


def _run_push(s):
    c, it = s["case"], s["integ"]
    p, n0, steps = c["order"], c["start"], c["steps"]
    it.pic_particles_write(*s["parts"])
    for r in range(p):
        it.pic_fields_upload(s["first"] + r, s["i0"][r], *s["levels"][r])
    counts = []
    if c["calls"] == "one":
        for r in range(p, p + steps):
            it.pic_fields_upload(s["first"] + r, s["i0"][r], *s["levels"][r])
        counts.append(_counts(it.pic_push_step(n0, steps, ok=OK)[0]))
    else:
        for j in range(steps):
            it.pic_fields_upload(n0 + j, s["i0"][p + j], *s["levels"][p + j])
            if c["carry"]:  # the coupled loop watches its counters
                it.pic_push_step(n0 + j, 1, ok=OK)
            else:
                it.pic_push_step(n0 + j, 1, want_stats=False)
        if not c["carry"]:
            counts.append(_counts(it.pic_stats_read()))
    it.pic_particles_read(*s["out"])
    if c["work"]:
        counts.append(it.work_read(s["done"]))
    return s["out"] + counts


def _run_noalloc(s):
    c = s["case"]
    for to, v in zip(s["out"], s["from"]):
        to.copy_(v)
    st = native.PicStepStats()
    code = native.lib().pic_push_mixed_noalloc(
        ctypes.byref(s["prm"]), c["n"], *[v.data_ptr() for v in s["out"]], s["E"], s["B"], s["i0"].ctypes.data,
        c["window"], c["start"], c["steps"], torch.cuda.current_stream().cuda_stream, ctypes.byref(st))
    if code not in OK:
        raise native.PicError(code, "pic_push_mixed_noalloc")
    return s["out"] + [_counts(st)]


def _run_predict(s):
    c = s["case"]
    if c["via"] == "fused":
        native.predict(s["integ"], s["net"], c["start"], s["pred"])
        return [s["pred"]]
    native.features(s["integ"], c["start"], s["phi"])
    s["net"].infer(s["phi"], s["pred"])
    return [s["pred"], s["phi"]]


def _run_train(s):
    c, net, b = s["case"], s["net"], s["case"]["batch"]
    net.set_params(s["params"])
    losses = [net.train_step(s["X"][q * b:(q + 1) * b], s["Y"][q * b:(q + 1) * b], c["lr"])
              for q in range(c["iters"])]
    return [np.array(losses, dtype=np.float32), net.get_params()]


def _run_batch(s):
    c, b = s["case"], s["batch"]
    wh = native.PIC_DEVICE
    b.particles_write(*s["parts"])
    for r, (E, B) in enumerate(s["levels"]):
        b.fields_upload(c["start"] - c["order"] + r, s["i0"][r], E, B)
    st = b.push_step(c["start"], c["steps"])
    b._chk(native.lib().pic_batch_particles_read(b.h, *[v.data_ptr() for v in s["out"]], wh))
    return s["out"] + [_counts(st)]


def _run_sc1d(s):
    c, loop = s["case"], s["loop"]
    loop.particles_write(*s["parts"])
    for l, lv in enumerate(s["levels"]):
        loop.fields_write(l - c["order"], *lv)
    st = loop.step(0, c["steps"])
    loop.particles_read(*s["out"])
    loop.fields_read(c["steps"], *s["fields"])
    return s["out"] + s["fields"] + [np.array(list(st.k_hist) + [st.substeps, st.n_star, st.clamped], dtype=np.int64)]


def _run_study(s):
    return native.study_run(s["cases"])


def work(c):
    """Bytes: inputs and results once.  Operations: ~60 of a Boris push and its two gathers, once
    per electron and step (the sub-steps beyond the first depend on the data)."""
    kind = c["kind"]
    if kind in ("push", "noalloc"):
        part = 33 + 32 if kind == "push" else 2 * 21
        lev = (c["order"] + c["steps"]) * c["window"] * 2 * (8 if kind == "push" else 4)
        return {"bytes": c["n"] * part + lev, "flops": 60 * c["n"] * c["steps"]}
    if kind == "predict":
        extra = 48 if c["via"] == "features" else 0
        return {"bytes": c["n"] * (22 + extra), "flops": 2 * 5120 * c["n"]}
    if kind == "train":
        n = c["batch"] * c["iters"]
        return {"bytes": 25 * n + 2 * 4 * 5128 * c["iters"], "flops": 6 * 5000 * n}
    if kind == "batch":
        mean = (c["largest"] - c["smallest"]) / math.log(c["largest"] / c["smallest"])
        n = c["ens"] * mean
        return {"bytes": n * 65 + (c["order"] + c["steps"]) * c["ens"] * c["window"] * 16, "flops": 60 * n * c["steps"]}
    if kind == "sc1d":
        n = c["cells"] * c["ppc"] * 0.9
        return {"bytes": n * 73 + (c["order"] + 2) * 24 * c["cells"], "flops": 100 * n * c["steps"]}
    q = _study_cases(c)
    n = sum(v["n_steps"] * v["n_electrons"] for v in q)
    return {"bytes": 400 * len(q), "flops": 200 * n}


# ---------------------------------------------------------------- the method in 64 bits

def _weights(p, is_e, theta):
    """The order-p Lagrange weights of the p + 1 levels at theta (a number)."""
    off = -0.5 if is_e else -1.0
    return [math.prod(((p - k) + off + theta) / (j - k) for k in range(p + 1) if k != j) for j in range(p + 1)]


class _Method:
    """Algorithm 1 on FP64 torch tensors: x, p, k_prev, dt, ... one value per electron (or numbers),
    `rows` lists of one level per entry, each a tuple of flat field arrays of n_ens x width values."""

    def __init__(self, order, field_time, psi, dt, dx, width, eid=None, k_max=7, work=None, lim=None):
        self.p, self.ft, self.psi, self.dt, self.dx = order, field_time, psi, dt, dx
        self.width, self.eid, self.k_max, self.work, self.lim = width, eid, k_max, work, lim
        self.iters = 0

    def gather(self, lv, i0, w, u, base):
        """Temporal sums at the two tent nodes of coordinate u, then the tent."""
        fl = torch.floor(u)
        j = fl.to(torch.int64)
        f0 = f1 = 0.0
        for l in range(self.p + 1):
            o = j - i0[l] + base
            f0 = f0 + w[l] * lv[l][o]
            f1 = f1 + w[l] * lv[l][o + 1]
        return f0 + (u - fl) * (f1 - f0)

    def step(self, S, fields, i0):
        """One macro step of S = dict(x, px, py, pz, k, lost[, work, dep]).  fields: name -> list of the
        p + 1 levels; i0: per level the window origins (a tensor over ensembles)."""
        dev = S["x"].device
        eid = self.eid
        on = (lambda v, q: v if not torch.is_tensor(v) or v.dim() == 0 else v[q])
        lo = torch.stack([v for v in i0]).max(0).values
        hi = torch.stack([v + self.width - 1 for v in i0]).min(0).values
        per = (lambda v, q: v[0] if eid is None else v[eid[q]])
        inv_dx = 1.0 / self.dx if not torch.is_tensor(self.dx) else 1.0 / self.dx
        every = torch.nonzero(~S["lost"]).flatten()

        def inside(u, q):
            if self.lim is not None:
                return (u >= self.lim[0]) & (u < self.lim[1])
            a, b = per(lo, q).double(), per(hi, q).double()
            return (u >= a) & (u < b) & (u - 0.5 >= a) & (u - 0.5 < b)

        s = S["x"][every] * on(inv_dx, every)
        ok = inside(s, every)
        S["lost"][every[~ok]] = True
        q = every[ok]
        u = S["x"][q] * on(inv_dx, q)
        org = [per(v, q) for v in i0]
        base = 0 if eid is None else eid[q] * self.width
        b0 = self.gather(fields["B"], org, _weights(self.p, False, 0.5), u - 0.5, base)
        g0 = torch.sqrt(1.0 + S["px"][q] ** 2 + S["py"][q] ** 2 + S["pz"][q] ** 2)
        psi = b0.abs() * on(self.dt, q) / (2.0 * g0)
        k = torch.zeros_like(q)
        for _ in range(self.k_max):
            up = psi > on(self.psi, q)
            k, psi = k + up, torch.where(up, 0.25 * psi, psi)
        for kk in range(self.k_max + 1):
            sel = q[k == kk]
            if sel.numel():
                self.cycle(S, fields, i0, sel, kk, inside, per, on, inv_dx)
        S["k"][q] = k

    def cycle(self, S, fields, i0, q, k, inside, per, on, inv_dx):
        m = 4 ** k
        x, px, py, pz = (S[v][q] for v in ("x", "px", "py", "pz"))
        dt = on(self.dt, q)
        h, h_old = dt / m, dt * torch.pow(0.25, S["k"][q].double())
        org = [per(v, q) for v in i0]
        base = 0 if self.eid is None else self.eid[q] * self.width
        live = torch.ones_like(x, dtype=torch.bool)
        inv = on(inv_dx, q)
        wk = torch.zeros_like(x)
        dep = S.get("dep")
        if dep is not None:
            dep["from"][q] = x
        for j in range(1, m + 1):
            u = x * inv
            now = live & inside(u, q)
            live = now
            u = torch.where(now, u, per(i0[-1], q).double() + 4.0) if self.lim is None else torch.where(now, u, self.lim[0] + 1.0)
            th = 0.5 + (j - 1) / m if self.ft == 0 else (j - 0.5) / m
            we, wb = _weights(self.p, True, th), _weights(self.p, False, th)
            ey = self.gather(fields["E"], org, we, u, base)
            bz = self.gather(fields["B"], org, wb, u - 0.5, base)
            half = 0.5 * (0.5 * (h_old + h) if j == 1 else h)
            dpx = -half * self.gather(fields["X"], org, we, u - 0.5, base) if "X" in fields else 0.0
            dpy = -ey * half
            vb = py / torch.sqrt(1.0 + px * px + py * py + pz * pz) if self.work else None
            mx, my = px + dpx, py + dpy
            tz = -bz * half / torch.sqrt(1.0 + mx * mx + my * my + pz * pz)
            ax, ay = mx + my * tz, my - mx * tz
            sz = 2.0 * tz / (1.0 + tz * tz)
            nx, ny = mx + ay * sz + dpx, my - ax * sz + dpy
            g = torch.sqrt(1.0 + nx * nx + ny * ny + pz * pz)
            px, py = torch.where(now, nx, px), torch.where(now, ny, py)
            if self.work:
                wk = wk + torch.where(now, -half * ey * (vb + ny / g), torch.zeros_like(g))
            if dep is not None:
                mid = (x + 0.5 * h * (nx / g)) * inv
                fl = torch.floor(mid)
                cw = torch.where(now, (ny / g) / m, torch.zeros_like(g)) * -dep["w"][q]
                dep["J"].index_add_(0, fl.long() + 2, cw * (1.0 - (mid - fl)))
                dep["J"].index_add_(0, fl.long() + 3, cw * (mid - fl))
            x = torch.where(now, x + h * (nx / g), x)
        self.iters += m
        S["x"][q], S["px"][q], S["py"][q] = x, px, py
        S["lost"][q[~live]] = True
        if self.work:
            S["done"][q] = S["done"][q] + wk


def _too_long(a0, dt, psi, steps, each=1.3e-3):
    """exact() would run past 20 s: `each` second per sub-step of the longest sub-cycles."""
    k = max(0, math.ceil(math.log(max(a0 * dt / (2.0 * psi), 1.0), 4.0)))
    return steps * (4 ** (min(k, 7) + 1) // 3) * each > 18.0


def _state(parts):
    x, px, py, pz = (v.clone() for v in parts[:4])
    return {"x": x, "px": px, "py": py, "pz": pz, "k": torch.zeros_like(x, dtype=torch.int64),
            "lost": torch.zeros_like(x, dtype=torch.bool), "done": torch.zeros_like(x)}


def exact(c, seed):
    kind = c["kind"]
    if kind in ("push", "noalloc"):
        few = c["n"] <= 4096  # on the host: less to launch per sub-step
        if _too_long(c["a0"], TWO_PI / c["res"], c["psi"], c["steps"], 6e-4 if few else 1.3e-3):
            return None
        dt, dx, i0, parts, levels = _push_inputs(c, seed)
        dev = "cpu" if few else DEV
        parts, levels = [v.to(dev) for v in parts], [[v.to(dev) for v in lv] for lv in levels]
        if kind == "noalloc":  # what the caller has: FP32 momenta and fields, the cell's offset in FP32
            sx = parts[0] * (1.0 / dx)
            parts = [(sx.floor() + (sx - sx.floor()).float().double()) * dx] + [v.float().double() for v in parts[1:]]
            levels = [[v.float().double() for v in lv] for lv in levels]
        S = _state(parts)
        M = _Method(c["order"], c["field_time"], c["psi"], dt, dx, c["window"], work=c["work"])
        org = [torch.tensor([int(v)], device=dev) for v in i0]
        for j in range(c["steps"]):
            r = slice(j, j + c["order"] + 1)
            M.step(S, {"E": [lv[0] for lv in levels[r]], "B": [lv[1] for lv in levels[r]]}, org[r])
        if kind == "noalloc":
            return [None, None] + [S[v] for v in ("px", "py", "pz")] + [None, None]
        counts = [None] * (0 if c["calls"] == "each" and c["carry"] else 1)
        return [S[v] for v in ("x", "px", "py", "pz")] + [None] + counts + ([S["done"]] if c["work"] else [])
    if kind == "predict":
        if c["via"] == "fused":
            return None  # classes
        dt, dx, i0, parts, levels = _push_inputs(c, seed)
        x, px, py, pz = parts
        f = []
        for name, w in ((0, _weights(c["order"], True, 1.5)), (1, _weights(c["order"], False, 1.5))):
            u = x / dx - 0.5 * name
            M = _Method(c["order"], 0, c["psi"], dt, dx, c["window"])
            f.append(torch.asinh(M.gather([lv[name] for lv in levels[:c["order"] + 1]],
                                          [int(v) for v in i0], w, u, 0).abs()))
        g = torch.sqrt(1.0 + px * px + py * py + pz * pz)
        return [None, torch.stack(f + [torch.asinh(v) for v in (px, py, pz)] + [torch.log(g)], dim=1)]
    if kind == "train":
        return _exact_train(c, seed)
    if kind == "batch":
        ens, eid, i0, parts, levels = _batch_inputs(c, seed)
        if _too_long(300.0, TWO_PI / 25, 0.003, c["steps"]):
            return None
        S = _state(parts)
        col = lambda n: torch.tensor([e[n] for e in ens], dtype=torch.float64, device=DEV)[eid]  # noqa: E731
        M = _Method(c["order"], 0, col("psi_max"), col("dt"), col("dx"), c["window"], eid=eid)
        org = [torch.as_tensor(v, device=DEV) for v in i0]
        for j in range(c["steps"]):
            r = slice(j, j + c["order"] + 1)
            M.step(S, {"E": [lv[0].flatten() for lv in levels[r]], "B": [lv[1].flatten() for lv in levels[r]]}, org[r])
        return [S[v] for v in ("x", "px", "py", "pz")] + [None, None]
    if kind == "sc1d":
        return _exact_sc1d(c, seed)
    return _exact_study(c, seed)


def _exact_train(c, seed):
    X, Y, packed = _train_inputs(c, seed)
    P = {k: torch.tensor(v, dtype=torch.float64, device=DEV, requires_grad=True)
         for k, v in native.unpack_params(packed).items()}
    names, losses = ("W1", "b1", "W2", "b2", "W3", "b3"), []
    m1, m2 = ({k: torch.zeros_like(v) for k, v in P.items()} for _ in range(2))
    for q in range(c["iters"]):
        x, y = (v[q * c["batch"]:(q + 1) * c["batch"]] for v in (X.double(), Y.long()))
        h = torch.relu(torch.relu(x @ P["W1"].T + P["b1"]) @ P["W2"].T + P["b2"])
        loss = torch.nn.functional.cross_entropy(h @ P["W3"].T + P["b3"], y)
        grads = torch.autograd.grad(loss, [P[k] for k in names])
        losses.append(float(loss))
        with torch.no_grad():
            for k, g in zip(names, grads):
                m1[k].mul_(0.9).add_(0.1 * g)
                m2[k].mul_(0.999).add_(0.001 * g * g)
                a, b = m1[k] / (1 - 0.9 ** (q + 1)), m2[k] / (1 - 0.999 ** (q + 1))
                P[k].sub_(c["lr"] * a / (b.sqrt() + 1e-8))
    return [np.array(losses), torch.cat([P[k].detach().flatten() for k in names])]


def _exact_sc1d(c, seed):
    wl, parts, levels = _sc1d_inputs(c, seed)
    if _too_long(c["a0"], wl.dt, c["psi"], c["steps"]):
        return None
    N, p, dt, dx, w = c["cells"], c["order"], wl.dt, wl.dx, parts[4]
    S = _state(parts)
    org = [torch.tensor([-2], device=DEV)] * (p + 1)
    r = dt / dx
    kap = (r - 1.0) / (r + 1.0)
    hist = [list(lv) for lv in levels]
    for _ in range(c["steps"]):
        M = _Method(p, c["field_time"], c["psi"], dt, dx, N + 5, lim=(0.5, N - 0.5))
        S["dep"] = {"w": w, "J": torch.zeros(N + 5, dtype=torch.float64, device=DEV), "from": S["x"].clone()}
        M.step(S, {"X": [h[0] for h in hist], "E": [h[1] for h in hist], "B": [h[2] for h in hist]}, org)
        J = S["dep"]["J"]
        # J_x at the faces from charge conservation: the change of charge to the left of each
        moved = torch.zeros(N + 5, dtype=torch.float64, device=DEV)
        for pos, sign in ((S["dep"]["from"], -1.0), (S["x"], 1.0)):
            u = pos / dx
            f = torch.floor(u)
            moved.index_add_(0, f.long() + 2, -sign * w * (1.0 - (u - f)))
            moved.index_add_(0, f.long() + 3, -sign * w * (u - f))
        X, E, B = hist[-1]
        F = -torch.cumsum(moved, 0)
        n = torch.arange(2, N + 3, device=DEV)
        e = torch.zeros_like(E)
        e[n] = E[n] - r * (B[n] - B[n - 1]) - dt * J[n]
        e[2] = E[3] + kap * (e[3] - E[2])
        e[N + 2] = E[N + 1] + kap * (e[N + 1] - E[N + 2])
        f = torch.arange(2, N + 2, device=DEV)
        b = torch.zeros_like(B)
        b[f] = B[f] - r * (e[f + 1] - e[f])
        hist = hist[1:] + [[X - F * dx, e, b]]
    return [S[v] for v in ("x", "px", "py", "pz")] + [None] + hist[-1] + [None]


def _exact_study(c, seed):
    r = np.random.Generator(np.random.PCG64(seed))
    cases = [dict(q, a0=q["a0"] * (1.0 + 1e-3 * r.random())) for q in _study_cases(c)]
    if sum(q["n_steps"] for q in cases) * 2.5 * 1.6e-4 > 18.0:
        return None
    got = []
    for q in cases:
        p, dt, n_e = q["order"], TWO_PI / q["res"], q["n_electrons"]
        dx = dt / 0.99
        xi0, sig = W.STUDY_XI0, W.STUDY_SIGMA

        def env(xi):
            return q["a0"] * np.exp(-((xi - xi0) ** 2) / (2.0 * sig * sig))

        def field(off, n, w, u):
            fl = np.floor(u)
            t = ((n - p + np.arange(p + 1)) + off)[:, None, None] * dt
            xi = t - np.stack([fl + off, fl + 1.0 + off])[None] * dx
            f = np.tensordot(w, -env(xi) * (np.cos(xi) - (xi - xi0) / sig ** 2 * np.sin(xi)), 1)
            return f[0] + (u - fl) * (f[1] - f[0])

        x, px, py = TWO_PI * np.arange(n_e) / n_e, np.zeros(n_e), np.zeros(n_e)
        h_old, wh = np.full(n_e, dt), np.array(_weights(p, False, 0.5))
        e_r, e_e, gm = (np.zeros(n_e), np.zeros(n_e), np.ones(n_e))
        g = np.ones(n_e)
        for n in range(q["n_steps"]):
            psi = np.abs(field(0.5, n, wh, x / dx - 0.5)) * dt / (2.0 * np.sqrt(1.0 + px * px + py * py))
            k = np.zeros(n_e, dtype=np.int64)
            for _ in range(7):
                up = psi > q["psi_max"]
                k, psi = k + up, np.where(up, 0.25 * psi, psi)
            h = dt / 4.0 ** k
            for kk in np.unique(k):
                s, m = k == kk, 4 ** int(kk)
                X, a, b = x[s], px[s], py[s]
                for j in range(1, m + 1):
                    th = 0.5 + (j - 1) / m
                    ey = field(0.0, n, np.array(_weights(p, True, th)), X / dx)
                    bz = field(0.5, n, np.array(_weights(p, False, th)), X / dx - 0.5)
                    half = 0.5 * (0.5 * (h_old[s] + h[s]) if j == 1 else h[s])
                    my = b - ey * half
                    tz = -bz * half / np.sqrt(1.0 + a * a + my * my)
                    ax, ay, sz = a + my * tz, my - a * tz, 2.0 * tz / (1.0 + tz * tz)
                    a, b = a + ay * sz, my - ax * sz - ey * half
                    gg = np.sqrt(1.0 + a * a + b * b)
                    X = X + h[s] * (a / gg)
                x[s], px[s], py[s], g[s] = X, a, b, gg
            h_old = h
            xi = (n + 1) * dt - 0.5 * h - (x - 0.5 * h * (px / g))
            g_th = 1.0 + 0.5 * (env(xi) * np.sin(xi)) ** 2
            e_r, e_e, gm = np.maximum(e_r, np.abs(g - px - 1.0)), np.maximum(e_e, np.abs(g - g_th) / g_th), np.maximum(gm, g)
        got.append({"eps_dephasing": float(e_r.max()), "eps_energy": float(e_e.max()), "gamma_max": float(gm.max()),
                    "eps_dephasing_first": float(e_r[0]), "eps_energy_first": float(e_e[0]),
                    "gamma_max_first": float(gm[0])})
    return got
