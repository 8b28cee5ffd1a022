"""Performance cases of the QED event generator: what users of the library run,
through its public entry points, over the range of sizes they run it at.

A case names an entry point (``kind``) and its sizes.  Inputs are made on the
GPU from the seed, with the recipes of ``paper_2008_10468_gb300/inputs.py``
(same populations, drawn by torch).  An event step changes its store in place,
so a pass first writes the momenta and types of the rows back, as a PIC code
does that hands over the particles it has pushed.  Children are appended in an
order that differs from run to run; a pass returns them ordered by id, in
buffers that hold as many as the store does (unused entries are 0).
"""
import math

import numpy as np
import torch

from paper_2008_10468_gb300 import qed

C_LIGHT, TAU_C = 299792458.0, 1.2880886664441626e-21   # m / s; hbar / (m c^2) in s
E_S = 1e-6 / (2.0 * math.pi * C_LIGHT * TAU_C)          # Schwinger field, code units at 1 um


def listed():
    return [
        # synchrotron functions: a tabulation by a user's script, and the sweep of
        # the benchmark; in binary64 (the accuracy of the paper's Table 1)
        {"name": "f1f2_4099", "kind": "f1f2", "n": 4099, "want": "both", "offset": 0},
        {"name": "f1f2_2p28", "kind": "f1f2", "n": 1 << 28, "want": "both", "offset": 0},
        {"name": "f1f2_f64_2p24", "kind": "f64", "n": 1 << 24},
        # per-cell sub-step counts of a large store (64 rows per cell)
        {"name": "plan_cells_2p24", "kind": "plan", "n": 1 << 24, "rows_per_cell": 64},
        # the global step with its cascade: a small store, where latency counts; the
        # electrons of the plain benchmark; the benchmark's clumped population
        {"name": "step_clumped_4133", "kind": "step", "n": 4133, "hot": 0.01, "rows_per_cell": 0},
        {"name": "step_uniform_1e5", "kind": "uniform", "n": 100000},
        {"name": "step_clumped_2p24", "kind": "step", "n": 1 << 24, "hot": 0.01,
         "rows_per_cell": 0},
        # the step with the Boris push before every draw
        {"name": "push_clumped_2p22", "kind": "push", "n": 1 << 22, "hot": 0.01,
         "rows_per_cell": 0},
        # the step on a store in page-locked host memory (a PIC code on the CPU)
        {"name": "host_clumped_2p20", "kind": "host", "n": 1 << 20, "hot": 0.01},
        # cascade batch: independent cells, one captured step with compaction and
        # drain of the low-chi photons (pools grow tenfold per step)
        {"name": "cascade_4096_cells", "kind": "cascade", "cells": 4096, "n_max": 16384},
        # the event-driven learned samplers in the step
        {"name": "sampler_clumped_2p22", "kind": "sampler", "n": 1 << 22, "hot": 0.01},
        # training of the emission sampler (forward, backward, Adam)
        {"name": "train_2p21", "kind": "train", "samples": 1 << 21, "batch": 2048},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["f1f2", "f64", "plan", "step", "step", "uniform", "push", "host",
                       "cascade", "sampler", "train"])
    if kind == "f1f2":
        return {"kind": kind, "n": _log_int(rng, 1000, 1 << 28),
                "want": rng.choice(["both", "both", "F1", "F2"]), "offset": rng.choice([0, 0, 1])}
    if kind == "f64":
        return {"kind": kind, "n": _log_int(rng, 1000, 1 << 24)}
    if kind == "plan":
        return {"kind": kind, "n": _log_int(rng, 1000, 1 << 24),
                "rows_per_cell": rng.choice([0, 1, 17, 64, 1000])}
    if kind in ("step", "push"):
        return {"kind": kind, "n": _log_int(rng, 500, 1 << (23 if kind == "step" else 22)),
                "hot": round(math.exp(rng.uniform(math.log(0.002), math.log(0.02))), 5),
                "rows_per_cell": rng.choice([0, 0, 64])}
    if kind == "uniform":
        return {"kind": kind, "n": _log_int(rng, 1000, 400000)}
    if kind == "host":
        return {"kind": kind, "n": _log_int(rng, 1000, 1 << 20), "hot": 0.01}
    if kind == "cascade":
        return {"kind": kind, "cells": _log_int(rng, 32, 4096), "n_max": rng.choice([1024, 16384])}
    if kind == "sampler":
        return {"kind": kind, "n": _log_int(rng, 10000, 1 << 22), "hot": 0.01}
    return {"kind": "train", "samples": _log_int(rng, 1 << 15, 1 << 21),
            "batch": rng.choice([1000, 2048, 4096, 8192])}


# --------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uniform(g, n):
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float64)


def _loguniform(g, n, lo, hi):
    return torch.exp(math.log(lo) + (math.log(hi) - math.log(lo)) * _uniform(g, n))


def _directions(g, n):
    mu = 2.0 * _uniform(g, n) - 1.0
    phi = 2.0 * math.pi * _uniform(g, n)
    s = torch.sqrt(torch.clamp(1.0 - mu * mu, min=0.0))
    return mu, s * torch.cos(phi), s * torch.sin(phi)


def _head_on(g, px, py, pz, eps, chi):
    """Crossed field met head-on: E = E0 e1, B = -E0 (n x e1), e1 at a random
    angle around n = p / |p|, E0 = chi E_s / (eps + |p|)."""
    p = torch.sqrt(px * px + py * py + pz * pz)
    nx, ny, nz = px / p, py / p, pz / p
    use_x = (nx.abs() < 0.9).double()
    ax, ay = use_x, 1.0 - use_x
    ux, uy, uz = ay * nz, -ax * nz, ax * ny - ay * nx
    un = torch.sqrt(ux * ux + uy * uy + uz * uz)
    ux, uy, uz = ux / un, uy / un, uz / un
    vx, vy, vz = ny * uz - nz * uy, nz * ux - nx * uz, nx * uy - ny * ux
    phi = 2.0 * math.pi * _uniform(g, p.numel())
    c, s = torch.cos(phi), torch.sin(phi)
    ex, ey, ez = c * ux + s * vx, c * uy + s * vy, c * uz + s * vz
    E0 = chi * E_S / (eps + p)
    return (E0 * ex, E0 * ey, E0 * ez, -E0 * (ny * ez - nz * ey), -E0 * (nz * ex - nx * ez),
            -E0 * (nx * ey - ny * ex))


def _fill(store, n, p, fields, types):
    for k, v in zip(("px", "py", "pz"), p):
        getattr(store, k)[:n] = v.float()
    for k, v in zip(("Ex", "Ey", "Ez", "Bx", "By", "Bz"), fields):
        getattr(store, k)[:n] = v.float()
    store.w[:n] = 1.0
    store.id[:n] = torch.arange(n, device="cuda")
    store.type[:n] = types
    store.count.fill_(n)


def _particles(g, n, capacity, gamma, chi, types):
    """Store of n rows with energies gamma, isotropic directions and head-on fields."""
    mx, my, mz = _directions(g, n)
    photon = types == qed.PHOTON
    pm = torch.where(photon, gamma, torch.sqrt(gamma * gamma - 1.0))
    p = [(pm * m).float().double() for m in (mx, my, mz)]
    p2 = p[0] * p[0] + p[1] * p[1] + p[2] * p[2]
    eps = torch.sqrt(torch.where(photon, p2, p2 + 1.0))
    store = qed.ParticleStore(capacity)
    _fill(store, n, p, _head_on(g, *p, eps, chi), types)
    return store


def _clumped(n, hot, seed, capacity):
    """25% e-, 25% e+, 50% photons; a contiguous block of the rows has chi in
    [10, 100], the rest in [1e-3, 1e-2]."""
    g = _gen(seed)
    r = _uniform(g, n)
    types = torch.where(r < 0.25, qed.ELECTRON, torch.where(r < 0.5, qed.POSITRON, qed.PHOTON))
    types = types.to(torch.uint8)
    n_hot = int(round(n * hot))
    h0 = (n - n_hot) // 2
    rows = torch.arange(n, device="cuda")
    is_hot = (rows >= h0) & (rows < h0 + n_hot)
    gamma = torch.where(is_hot, _loguniform(g, n, 3e3, 3e4), _loguniform(g, n, 1e2, 1e3))
    chi = torch.where(is_hot, _loguniform(g, n, 10.0, 100.0), _loguniform(g, n, 1e-3, 1e-2))
    return _particles(g, n, capacity, gamma, chi, types)


def _uniform_electrons(n, seed, capacity):
    """Electrons with gamma in [1e2, 1e4] and chi in [0.1, 10], log-uniform."""
    g = _gen(seed)
    gamma, chi = _loguniform(g, n, 1e2, 1e4), _loguniform(g, n, 0.1, 10.0)
    types = torch.zeros(n, device="cuda", dtype=torch.uint8)
    return _particles(g, n, capacity, gamma, chi, types)


def _cell_sizes(cells, n_max):
    """Power-law particle counts (exponent -1.5) on [1, n_max]: one per quantile."""
    u = (np.arange(cells) + 0.5) / cells
    a = -0.5
    return np.clip(np.floor((1.0 + u * (float(n_max) ** a - 1.0)) ** (1.0 / a)), 1,
                   n_max).astype(np.int64)


def _cascade(cells, n_max, seed, capacity):
    """Electrons of independent cells, one crossed field E y, B z per cell; the
    cells' chi (for gamma 1e3 moving against the field) log-uniform in [1e-2, 50]."""
    g = _gen(seed)
    counts = torch.from_numpy(_cell_sizes(cells, n_max)).cuda()
    chi = 1e-2 * 5e3 ** ((torch.randperm(cells, generator=g, device="cuda") + 0.5) / cells).double()
    E0 = torch.repeat_interleave(chi * E_S / 2e3, counts)
    n = E0.numel()
    gamma = _loguniform(g, n, 1e2, 1e4)
    pm = torch.sqrt(gamma * gamma - 1.0)
    zero = torch.zeros_like(E0)
    store = qed.ParticleStore(capacity)
    _fill(store, n, [pm * m for m in _directions(g, n)], (zero, E0, zero, zero, zero, E0),
          torch.zeros(n, device="cuda", dtype=torch.uint8))
    return store, n


def _points(n, seed, dtype):
    y = 1e-4 * torch.exp(math.log(50.0 / 1e-4) * _uniform(_gen(seed), n))
    return torch.clamp(y, 1e-4, 50.0).to(dtype)


def _cells(n, rows_per_cell):
    """Cell index per row (rows grouped by cell) and the number of cells."""
    return ((torch.arange(n, device="cuda") // rows_per_cell).to(torch.int32),
            -(-n // rows_per_cell))


def _cascade_capacity(n):
    return min(1 << 26, max(1 << 22, 256 * n))


def prepare(case, seed):
    k = case["kind"]
    s = {"case": case}
    if k == "f1f2":
        n, off = case["n"], case["offset"]
        y = torch.empty(n + off, device="cuda")
        y[off:] = _points(n, seed, torch.float32)
        s["y"] = y[off:]
        s["F1"] = torch.empty(n + off, device="cuda")[off:] if case["want"] != "F2" else None
        s["F2"] = torch.empty(n + off, device="cuda")[off:] if case["want"] != "F1" else None
        s["ctx"] = qed.Context(seed=seed)
        return s
    if k == "f64":
        s["y"] = _points(case["n"], seed, torch.float64)
        s["F1"], s["F2"] = torch.empty_like(s["y"]), torch.empty_like(s["y"])
        return s
    if k == "train":
        s["ctx"] = qed.Context(seed=seed, sampler="event")
        s["seed"] = seed
        r = np.random.default_rng(seed)
        fan = np.full(qed.SAMPLER_PARAMS, 64.0)
        fan[:192] = 2.0
        s["init"] = (r.uniform(-1.0, 1.0, qed.SAMPLER_PARAMS) / np.sqrt(fan)).astype(np.float32)
        return s
    if k == "cascade":
        cap = _cascade_capacity(int(_cell_sizes(case["cells"], case["n_max"]).sum()))
        store, n = _cascade(case["cells"], case["n_max"], seed, cap)
        s["ctx"] = qed.Context(seed=seed, drain_chi=0.05)
        s["ctx"].graph_capture(store, 0, 1)
        s["rows"] = {f: getattr(store, f)[:n].clone() for f in qed.FLOAT_FIELDS + ("id", "type")}
    else:
        n = case["n"]
        if k == "uniform":
            store = _uniform_electrons(n, seed, 24 * n + 8192)
            s["ctx"] = qed.Context(seed=seed, process_mask=qed.PROC_EMISSION)
        else:
            cap = n if k == "plan" else (3 if case["hot"] <= 0.01 else 5) * n + 8192
            store = _clumped(n, case.get("hot", 0.01), seed, cap)
            s["ctx"] = qed.Context(seed=seed, sampler="event" if k == "sampler" else False,
                                   sampler_max_err=1e-2)
        if k == "sampler":
            # the weights such a program keeps: both networks, a short training
            for process in (qed.PROC_EMISSION, qed.PROC_PAIR):
                s["ctx"].sampler_process(process)
                s["ctx"].sampler_train(20081051, 1 << 22, batch=2048, lr=3e-3)
                s["ctx"].sampler_evaluate()
        if case.get("rows_per_cell"):
            s["cell"], s["ncells"] = _cells(n, case["rows_per_cell"])
        if k == "plan":
            s["chi"] = torch.empty(n, device="cuda")
            s["N"] = torch.empty(n if "cell" not in s else s["ncells"], device="cuda",
                                 dtype=torch.int32)
        s["rows"] = {f: getattr(store, f)[:n].clone() for f in ("px", "py", "pz", "type")}
    s["store"], s["n"] = store, n
    if k != "plan":
        room = store.capacity - n
        s["child"] = {"id": torch.zeros(room, device="cuda", dtype=torch.int64),
                      "type": torch.zeros(room, device="cuda", dtype=torch.uint8),
                      "fields": torch.zeros(len(qed.FLOAT_FIELDS), room, device="cuda")}
        s["order"] = torch.empty(room, device="cuda", dtype=torch.int64)
    if k == "host":
        h = qed.HostStore(store.capacity)
        for f in qed.FLOAT_FIELDS + ("id", "type"):
            getattr(h, f)[:n].copy_(getattr(store, f)[:n])
        s["rows"] = {f: t.cpu().pin_memory() for f, t in s["rows"].items()}
        s["store"] = h
    return s


# --------------------------------------------------------------------------
# One pass
# --------------------------------------------------------------------------
STATS = ("status", "substeps", "emissions", "pairs", "children", "guard_hits", "plans", "max_N",
         "count")


def _out(s, stats):
    """Momenta and types of the rows given, the rows appended in order of their
    ids, and the step's counts."""
    store, child, n, m = s["store"], s["child"], s["n"], stats["count"]
    out = {f: getattr(store, f)[:n] for f in ("px", "py", "pz", "type")}
    order = s["order"][:m - n]
    torch.sort(store.id[n:m].cuda(non_blocking=True), out=(child["id"][:m - n], order))
    torch.index_select(store.type[n:m].cuda(non_blocking=True), 0, order, out=child["type"][:m - n])
    fields = [getattr(store, f)[n:m] for f in qed.FLOAT_FIELDS]
    torch.index_select(torch.stack([f.cuda(non_blocking=True) for f in fields]), 1, order,
                       out=child["fields"][:, :m - n])
    out["child"] = child
    out["stats"] = [int(stats[k]) for k in STATS]
    return out


def run(s):
    case = s["case"]
    k = case["kind"]
    if k == "f1f2":
        s["ctx"].synchrotron_F1F2(s["y"], s["F1"], s["F2"])
        return [s["F1"], s["F2"]]
    if k == "f64":
        qed.synchrotron_F1F2_f64(s["y"], s["F1"], s["F2"])
        return [s["F1"], s["F2"]]
    ctx = s["ctx"]
    if k == "train":
        ctx.sampler_load(s["init"])
        loss = ctx.sampler_train(s["seed"], case["samples"], batch=case["batch"], lr=3e-3)
        return {"params": ctx.sampler_save(), "loss": np.float32(loss)}
    store, n = s["store"], s["n"]
    if k == "plan":
        if "cell" in s:
            return {"N": ctx.plan_cells(store, n, s["cell"], s["ncells"], s["N"])}
        ctx.plan(store, n, s["chi"], s["N"])
        return {"chi": s["chi"], "N": s["N"]}
    for f, t in s["rows"].items():
        getattr(store, f)[:n].copy_(t)
    if k == "host":
        store.count = n
        return _out(s, ctx.event_step_host(store, 0))
    store.count.fill_(n)
    if k == "cascade":
        ctx.graph_launch()
        stats = ctx.graph_read_stats()[0]
        for t in s["child"].values():   # each launch is another step, with other counts
            t[..., stats["count"] - n:].zero_()
        out = _out(s, stats)
        out["spectrum"] = ctx.read_spectrum(reset=True)
        return out
    if "cell" in s:
        step = ctx.event_step_push_cells if k == "push" else ctx.event_step_cells
        stats = step(store, 0, s["cell"], s["ncells"])
    else:
        stats = ctx.event_step(store, 0, push=k == "push")
    return _out(s, stats)


# --------------------------------------------------------------------------
# What a pass cannot do without
# --------------------------------------------------------------------------
# per row of the populations (means): sub-steps and children of one step
PER_ROW = {"step": (6140.0, 37.8), "push": (2160.0, 14.0), "host": (6140.0, 37.8),
           "sampler": (6140.0, 37.8), "uniform": (1030.0, 9.5), "cascade": (11300.0, 49.0)}
ROW, CHANGED = 49, 13          # bytes of a row; of its momentum and type
SUBSTEP_OPS = 45               # half a Philox block and its test
EVENT_OPS = 2 * 8577           # one network evaluation


def work(case):
    k = case["kind"]
    if k == "f1f2":
        outs = 2 if case["want"] == "both" else 1
        return {"bytes": 4 * (1 + outs) * case["n"], "flops": 14 * outs * case["n"]}
    if k == "f64":
        return {"bytes": 24 * case["n"], "flops": 48 * case["n"]}
    if k == "train":
        return {"bytes": 8 * qed.SAMPLER_PARAMS, "flops": 6 * qed.SAMPLER_PARAMS * case["samples"]}
    if k == "plan":
        # type, momentum and fields of a row; chi and N, or the cell index
        return {"bytes": (37 + (4 if case["rows_per_cell"] else 8)) * case["n"],
                "flops": 100 * case["n"]}
    if k == "cascade":
        n, hot = int(_cell_sizes(case["cells"], case["n_max"]).sum()), 1.0
    else:
        n, hot = case["n"], case.get("hot", 1.0)
    sub, kids = PER_ROW[k]
    # the sampler draws the sub-steps to an event at once: its work is the events
    ops = EVENT_OPS * 0.95 * kids if k == "sampler" else SUBSTEP_OPS * sub
    return {"bytes": (ROW + CHANGED) * n + ROW * kids * hot * n, "flops": ops * hot * n}


# --------------------------------------------------------------------------
# The same in 64 bits
# --------------------------------------------------------------------------
def _FG64(y):
    """F = y int exp(-y cosh t) cosh(5t/3) / cosh t dt and G = y int exp(-y cosh t)
    cosh(2t/3) dt over t > 0 (trapezoid rule, which converges geometrically)."""
    h = 0.1
    F, G = torch.empty_like(y), torch.empty_like(y)
    for i in range(0, y.numel(), 1 << 24):
        x = y[i:i + (1 << 24)]
        f, g = torch.zeros_like(x), torch.zeros_like(x)
        for j in range(150):
            t = j * h
            w = h if j else 0.5 * h
            e = torch.exp(x * -math.cosh(t))
            f.add_(e, alpha=w * math.cosh(5.0 * t / 3.0) / math.cosh(t))
            g.add_(e, alpha=w * math.cosh(2.0 * t / 3.0))
        F[i:i + (1 << 24)], G[i:i + (1 << 24)] = x * f, x * g
    return F, G


def _chi64(store, n):
    """chi = sqrt((eps E + p x B)^2 - (p . E)^2) / E_s of rows [0, n)."""
    px, py, pz, Ex, Ey, Ez, Bx, By, Bz = (getattr(store, f)[:n].double()
                                          for f in qed.FLOAT_FIELDS[:9])
    p2 = px * px + py * py + pz * pz
    eps = torch.sqrt(torch.where(store.type[:n] == qed.PHOTON, p2, p2 + 1.0))
    ax = eps * Ex + py * Bz - pz * By
    ay = eps * Ey + pz * Bx - px * Bz
    az = eps * Ez + px * By - py * Bx
    pe = px * Ex + py * Ey + pz * Ez
    return torch.sqrt(torch.clamp(ax * ax + ay * ay + az * az - pe * pe, min=0.0)) / E_S


def exact(case, seed):
    """64-bit values of the synchrotron functions and of chi.  The events of a step
    and the trained weights follow from every rounding before them: no such value."""
    k = case["kind"]
    if k in ("f1f2", "f64"):
        F, G = _FG64(_points(case["n"], seed, torch.float32 if k == "f1f2" else torch.float64)
                     .double())
        want = case.get("want", "both")
        return [F if want != "F2" else None, G if want != "F1" else None]
    if k == "plan" and not case["rows_per_cell"]:
        s = prepare(case, seed)
        return {"chi": _chi64(s["store"], s["n"]), "N": None}
    return None
