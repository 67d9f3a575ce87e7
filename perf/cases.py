"""What this framework is measured on: the work its users have it do, through its public entry points.

Kinds of case:
  steps   a discharge (or a batch) advanced by a number of time steps, then its cycle-averaged moments
          (with the discharge current), the field and, where configured, the kinetic diagnostics read out:
          the loop of every production run, from a small warm-start family member to the beyond-L2 discharge;
  state   the whole particle state restored from pinned host arrays, one step, the state and the moments read
          back: a host code that couples to the library every step;
  train   steps of Adam on the warm-start network, then its parameters;
  predict the warm-start network's forward pass;
  sort    the allocation-free stable sort of a caller-owned particle store.

Discharges, time steps and table grids are those of the package's named workloads and warm-start family, at
their own and other sizes.
"""
from __future__ import annotations

import ctypes as C
import functools
import math

import numpy as np
import torch

from paper_1608_04601_gb300 import _native as NV
from paper_1608_04601_gb300 import mlp, pic, warmstart
from paper_1608_04601_gb300 import xsections as X
from paper_1608_04601_gb300.workloads import Discharge

# What a discharge needs beyond its sizes: (gas, pressure Pa, gap m, voltage V, initial density m^-3, steps per
# rf period, secondary emission, table's last energy eV, table step eV).
REGIMES = {
    "he_family": ("he", 26.0, 0.022, 380.0, 4e14, 400, 0.0, 800.0, 1e-2),  # the warm-start family's middle
    "ar_10Pa": ("ar", 10.0, 0.025, 300.0, 4e15, 2000, 0.0, 1000.0, 1e-3),
    "he_80Pa": ("he", 80.0, 0.05, 150.0, 4e14, 4000, 0.1, 2000.0, 1e-3),  # secondary electrons
}
WARM_NET = "-".join(str(s) for s in warmstart.SIZES)


def _steps(name, regime, cells, n_e, n_i, steps, **kw):
    c = dict(kind="steps", regime=regime, cells=cells, n_e=n_e, n_i=n_i, steps=steps, batch=1, spread=1.0,
             precision="fp32", sort_every=16, graph=False, leapfrog=False, sample_every=0)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one discharge of the warm-start family on its own: the smallest run, an rf period as one CUDA graph
        _steps("one small discharge, graph", "he_family", 128, 20000, 20000, 400, sort_every=8, graph=True),
        # a run with the library's defaults (no sort, no graph) at odd sizes
        _steps("defaults, odd sizes", "he_family", 101, 150001, 133337, 80, sort_every=0),
        # the benchmark discharge: 1e6 + 1e6, 512 cells
        _steps("benchmark discharge", "ar_10Pa", 512, 1000000, 1000000, 64),
        # the same on the FP64 path
        _steps("benchmark discharge, fp64", "ar_10Pa", 512, 1000000, 1000000, 32, precision="fp64"),
        # the leapfrog variant with the kinetic diagnostics' EEDF samples every 8 steps, ragged sizes
        _steps("leapfrog, diagnostics", "ar_10Pa", 777, 611953, 588235, 64, leapfrog=True, sample_every=8),
        # a discharge beyond L2: 1.2e7 + 1.2e7, 2048 cells, secondary electrons
        _steps("large discharge", "he_80Pa", 2048, 12000000, 12000000, 24),
        # training data of the warm start: 64 family members in one launch per step, an rf period
        _steps("family batch", "he_family", 128, 20000, 20000, 400, batch=64, sort_every=8, graph=True),
        # a parameter scan with uneven particle numbers, 3e4 .. 1.3e6 a species
        _steps("uneven batch", "ar_10Pa", 512, 200000, 200000, 32, batch=16, spread=6.3),
        # state up and down every step over the host link
        {"name": "state up and down", "kind": "state", "regime": "ar_10Pa", "cells": 512, "n_e": 1000000,
         "n_i": 1000000, "sort_every": 16},
        # the warm-start network: training steps at its batch, and predictions for a handful of discharges
        {"name": "network training", "kind": "train", "sizes": WARM_NET, "batch": 256, "steps": 20},
        {"name": "network prediction", "kind": "predict", "sizes": WARM_NET, "batch": 24},
        # the sort of a caller-owned store a few steps after its last sort
        {"name": "caller-owned sort", "kind": "sort", "n": 1000000, "cells": 512, "precision": "fp32"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["steps"] * 6 + ["state", "train", "predict", "sort"])
    if kind == "steps":
        regime = rng.choice(sorted(REGIMES))
        spp = REGIMES[regime][5]
        cells = _log(rng, 32, 256) if spp == 400 else _log(rng, 200, 1000) if spp == 2000 else _log(rng, 600, 4096)
        batch = rng.choice([1, 1, 1, _log(rng, 2, 24)])
        n = _log(rng, 1e4, (4e5 if spp == 400 else 4e6) / (batch if batch > 1 else 1))
        graph = spp == 400 and n * batch <= 400000 and rng.random() < 0.6
        steps = spp if graph else max(8, min(200, int(1.2e8 / (n * batch))))
        return _steps(None, regime, cells, n, max(1000, int(n * rng.uniform(0.8, 1.2))), steps, batch=batch,
                      spread=rng.choice([1.0, 3.0]) if batch > 1 else 1.0,
                      precision=rng.choice(["fp32", "fp32", "fp32", "fp64"]), sort_every=rng.choice([0, 8, 16, 16]),
                      graph=graph, leapfrog=rng.random() < 0.25, sample_every=rng.choice([0, 0, 0, 8, 16]))
    if kind == "state":
        regime = rng.choice(["he_family", "ar_10Pa"])
        n = _log(rng, 1e4, 4e5 if regime == "he_family" else 1.5e6)
        return {"kind": "state", "regime": regime, "cells": 100 if regime == "he_family" else _log(rng, 200, 1000),
                "n_e": n, "n_i": int(n * rng.uniform(0.8, 1.2)), "sort_every": rng.choice([0, 16])}
    if kind == "sort":
        return {"kind": "sort", "n": _log(rng, 1000, 1.9e6), "cells": _log(rng, 16, 2000),
                "precision": rng.choice(["fp32", "fp32", "fp64"])}
    hidden = rng.choice([1, 2, 4])
    width = rng.choice([_log(rng, 48, 1024), 256, 512])
    sizes = "-".join(str(s) for s in [rng.randint(3, 12)] + [width] * hidden + [rng.choice([3 * warmstart.NPTS, 300])])
    batch = _log(rng, 1, 1024)
    if kind == "predict":
        return {"kind": kind, "sizes": sizes, "batch": batch}
    return {"kind": kind, "sizes": sizes, "batch": batch, "steps": 20}


# ---- states ---------------------------------------------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _gas(name, eps_max, de):
    return X.by_name(name, eps_max_eV=eps_max, de_eV=de)


def _counts(case):
    """(electrons, ions) of every discharge of the batch: `spread` apart, geometrically."""
    b = case.get("batch", 1)
    f = [case.get("spread", 1.0) ** (2.0 * i / (b - 1) - 1.0) if b > 1 else 1.0 for i in range(b)]
    return [(max(1, round(case["n_e"] * x)), max(1, round(case["n_i"] * x))) for x in f]


def _simulation(case, seed):
    """The discharges of a case, loaded homogeneously; stores with room for the growth of a long run."""
    gas, p, gap, V, n_init, spp, gamma, eps_max, de = REGIMES[case["regime"]]
    ds = []
    for i, (ne, ni) in enumerate(_counts(case)):
        # pressure and voltage vary a little over a batch, as in a parameter scan
        ds.append(Discharge("case", gas, gap, p * (1.0 + 0.004 * i), V * (1.0 + 0.003 * i), case["cells"], spp, ne, ni,
                            n_init, gamma_see=gamma, seed=seed, discharge_id=i))
    sim = pic.Simulation(_gas(gas, eps_max, de), ds, seed=seed, precision=case.get("precision", "fp32"),
                         sort_every=case["sort_every"], use_graph=case.get("graph", False),
                         capacity=[d.capacity(1.25 if d.n_e0 > 4000000 else 2.0 if d.n_e0 > 1000000 else 4.0) for d in ds],
                         leapfrog=case.get("leapfrog", False))
    if case.get("sample_every"):
        sim.set_diagnostics(period_steps=spp, phase_step=1, sample_every=case["sample_every"], eedf_bins=200,
                            eedf_de_eV=0.5, fast_eV=V / 4)
    return sim


def _weights(sizes, seed):
    """Glorot-uniform weights and small biases, in the layout of the network's parameters."""
    rng = np.random.default_rng(seed)
    out = []
    for i, o in zip(sizes[:-1], sizes[1:]):
        a = math.sqrt(6.0 / (i + o))
        out += [rng.uniform(-a, a, i * o), rng.normal(0.0, 0.02, o)]
    return np.concatenate(out).astype(np.float32)


def _net_data(case, seed):
    """Weights, inputs of order one and smooth profile targets, as float32 arrays."""
    sizes = [int(s) for s in case["sizes"].split("-")]
    rng = np.random.default_rng(seed + 7)
    x = rng.uniform(-1.0, 1.0, (case["batch"], sizes[0])).astype(np.float32)
    s = np.linspace(0.0, 1.0, sizes[-1])
    t = (1.0 + 0.5 * x[:, :1]) * np.sin(np.pi * s) + 0.3 * x[:, 1:2] * np.cos(2 * np.pi * s) + 0.2 * x[:, 2:3]
    return sizes, _weights(sizes, seed), x, t.astype(np.float32)


def _sort_data(case, seed):
    """A store some steps after a sort: slots in cell order but for a shift of a few cells."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n, cells = case["n"], case["cells"]
    real = torch.float32 if case["precision"] == "fp32" else torch.float64
    base = torch.sort(torch.randint(0, cells, (n,), generator=g, device="cuda")).values
    shift = torch.randn(n, generator=g, device="cuda") * 3.0
    c = (base + shift.round().to(torch.int64)).clamp(0, cells - 1).to(torch.int32)
    return c, torch.randn((n, 4), generator=g, device="cuda", dtype=real)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "steps":
        return {"case": case, "sim": _simulation(case, seed)}
    if kind == "state":
        sim = _simulation(case, seed)
        if case["sort_every"]:
            sim.sort()
        host = []
        for sp in (0, 1):  # pinned arrays the host program keeps, with the state it holds
            cap = int(1.5 * case["n_i" if sp else "n_e"]) + 64
            a = {"c": torch.zeros(cap, dtype=torch.int32, pin_memory=True).numpy()}
            a.update({k: torch.zeros(cap, dtype=torch.float32, pin_memory=True).numpy() for k in ("f", "vx", "vy", "vz")})
            host.append(a)
        now = [sim.get_state(0, sp, out=host[sp]) for sp in (0, 1)]
        return {"case": case, "sim": sim, "host": host, "now": now}
    if kind in ("train", "predict"):
        sizes, w, x, t = _net_data(case, seed)
        net = mlp.MLP(sizes, max_batch=case["batch"], seed=1)
        net.set_params(w)
        return {"case": case, "net": net, "x": torch.from_numpy(x).cuda(), "t": torch.from_numpy(t).cuda()}
    c, r = _sort_data(case, seed)
    return {"case": case, "c": c, "r": r, "c_out": torch.empty_like(c), "r_out": torch.empty_like(r)}


# ---- one pass -------------------------------------------------------------------------------------------------

_MOMENTS = ("n_e", "n_i", "mean_eps", "count", "absorbed", "flux", "surface_charge", "J_amp", "J_last")


def _read_moments(sim):
    ms = [sim.moments(d) for d in range(len(sim.N))]
    return {k: np.stack([np.asarray(m[k]) for m in ms]) for k in _MOMENTS}


def _run_steps(s):
    case, sim = s["case"], s["sim"]
    sim.step(case["steps"])
    out = _read_moments(sim)
    if case["batch"] == 1:
        out["E"], out["E64"], out["phi"] = sim.get_field(0)
    if case["sample_every"]:
        ds = [sim.diagnostics(d) for d in range(case["batch"])]
        out["diagnostics"] = {k: np.stack([np.asarray(d[k]) for d in ds]) for k in ds[0]}
    return out


def _run_state(s):
    sim = s["sim"]
    for sp in (0, 1):
        sim.set_state(0, sp, s["now"][sp])
    sim.step(1)
    s["now"] = [sim.get_state(0, sp, out=s["host"][sp]) for sp in (0, 1)]
    return {"moments": _read_moments(sim), "electrons": s["host"][0], "ions": s["host"][1]}


def run(state):
    kind = state["case"]["kind"]
    if kind == "steps":
        return _run_steps(state)
    if kind == "state":
        return _run_state(state)
    if kind == "predict":
        return state["net"].forward(state["x"])
    if kind == "train":
        net, n = state["net"], state["case"]["steps"]
        for _ in range(n - 1):
            net.train_step(state["x"], state["t"], 1e-4, sync=False)
        loss = net.train_step(state["x"], state["t"], 1e-4)
        return {"loss": loss, "params": net.get_params()}
    c, r = state["c"], state["r"]
    code = pic.FP32 if state["case"]["precision"] == "fp32" else pic.FP64
    NV.check(NV.lib().pic_sort_noalloc(
        C.c_void_p(c.data_ptr()), C.c_void_p(r.data_ptr()), C.c_void_p(state["c_out"].data_ptr()),
        C.c_void_p(state["r_out"].data_ptr()), c.numel(), state["case"]["cells"], code,
        C.c_void_p(torch.cuda.current_stream().cuda_stream)))
    return {"c": state["c_out"], "records": state["r_out"]}


# ---- what a pass cannot do without ----------------------------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind in ("steps", "state"):
        # each particle's record (cell, offset, three velocities) read and written once a step; about 60
        # operations each (gather, two kicks, energy, drift, charge and energy split)
        rec = 36 if case.get("precision") == "fp64" else 20
        particle_steps = sum(a + b for a, b in _counts(case)) * case.get("steps", 1)
        scale = 4 if kind == "state" else 2  # state: up and down over the host link as well
        return {"bytes": scale * rec * particle_steps, "flops": 60 * particle_steps}
    if kind == "sort":
        rec = 20 if case["precision"] == "fp32" else 36
        return {"bytes": 2 * rec * case["n"], "flops": 0}
    sizes = [int(s) for s in case["sizes"].split("-")]
    w = sum(i * o for i, o in zip(sizes[:-1], sizes[1:]))
    p, b = w + sum(sizes[1:]), case["batch"]
    if kind == "predict":  # BF16 weights read, inputs and outputs in FP32
        return {"bytes": 2 * w + 4 * b * (sizes[0] + sizes[-1]), "flops": 2 * b * w}
    first = sizes[0] * sizes[1]
    # three products a layer (the first layer has no input gradient); Adam reads and writes the FP32 weights and
    # two moments
    return {"bytes": case["steps"] * (24 * p + 4 * w + 4 * b * (sizes[0] + sizes[-1])),
            "flops": case["steps"] * 2 * b * (3 * w - first)}


# ---- the same in 64 bits --------------------------------------------------------------------------------------

def _forward64(p, sizes, x):
    ys, o = [x], 0
    for l, (i, n) in enumerate(zip(sizes[:-1], sizes[1:])):
        w, b = p[o:o + i * n].reshape(n, i), p[o + i * n:o + i * n + n]
        o += i * n + n
        z = ys[-1] @ w.T + b
        ys.append(np.tanh(z) if l + 2 < len(sizes) else z)
    return ys


def _loss_grad64(p, sizes, x, t):
    ys = _forward64(p, sizes, x)
    d = ys[-1] - t
    loss, g, grads, o = float(np.mean(d * d)), 2.0 * d / d.size, [], p.size
    for l in range(len(sizes) - 2, -1, -1):
        i, n = sizes[l], sizes[l + 1]
        o -= i * n + n
        grads[:0] = [(g.T @ ys[l]).ravel(), g.sum(0)]
        if l:
            g = (g @ p[o:o + i * n].reshape(n, i)) * (1.0 - ys[l] ** 2)
    return loss, np.concatenate(grads)


def exact(case, seed):
    kind = case["kind"]
    if kind == "sort":
        c, r = _sort_data(case, seed)
        c, at = torch.sort(c, stable=True)
        return {"c": c, "records": r[at].double()}
    if kind in ("steps", "state"):
        # no such value: every particle's collisions, cells and fates are decided in the path's own precision,
        # and one decision the other way changes every random stream after it
        return None
    sizes, w, x, t = _net_data(case, seed)
    p, x, t = w.astype(np.float64), x.astype(np.float64), t.astype(np.float64)
    if kind == "predict":
        return torch.from_numpy(_forward64(p, sizes, x)[-1])
    m, v = np.zeros_like(p), np.zeros_like(p)
    for k in range(1, case["steps"] + 1):
        loss, g = _loss_grad64(p, sizes, x, t)
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        p = p - 1e-4 * (m / (1.0 - 0.9 ** k)) / (np.sqrt(v / (1.0 - 0.999 ** k)) + 1e-8)
    return {"loss": loss, "params": p}
