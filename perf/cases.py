"""The workloads by which the speed of this framework is judged.

Each case is one pass through the public entry points (`UniformRun`, `AMRRun`, `Tagger`) over the range that
its users have: uniform grids from one 64 x 64 patch to 4096 x 4096 cells, adaptive forests with a fixed and
with a changing set of leaves, the learned tagger's inference and training, variable-velocity advection, and a
state kept in host memory.  Sizes are those of the configurations, the benchmark and the tests, or odd ones.

Outputs are the degrees of freedom that a patch owns (views of the state's own buffers, no copies), and beside
them tags, gradients and weights.  `exact` restates a step in plain 64-bit torch.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2205_07572_gb300 import af, tune
from paper_2205_07572_gb300.amr import AMRRun, Forest, regrid_arrays
from paper_2205_07572_gb300.tagger import Tagger
from paper_2205_07572_gb300.uniform import UniformRun

G = 2            # ghost layers
PREC = {"f32": af.F32, "f64": af.F64}
FIELD = {"const": None, "solid": af.FIELD_SOLID_BODY, "swirl": af.FIELD_SWIRL}
CFL = 0.4


def listed():
    return [
        # the smallest call: one 64 x 64 patch, FP64 advection with a = (1, 0.5) (configuration 1)
        {"name": "advection_f64_64", "kind": "uniform", "eq": "advection", "prec": "f64", "field": "const",
         "n": 64, "px": 1, "py": 1, "a": 1.0, "b": 0.5, "tune": False},
        # patches of an odd size on a ragged grid, the library's default tiling
        {"name": "advection_f32_odd", "kind": "uniform", "eq": "advection", "prec": "f32", "field": "const",
         "n": 23, "px": 61, "py": 53, "a": 1.0, "b": -0.7, "tune": False},
        # acoustics on 512 x 512 cells in 32 x 32 patches (configuration 2): a step at a time, in cache
        {"name": "acoustics_f32_512", "kind": "uniform", "eq": "acoustics", "prec": "f32", "field": "const",
         "n": 32, "px": 16, "py": 16, "a": 0.0, "b": 0.0, "tune": True},
        # the same in FP64, the other precision of that configuration
        {"name": "acoustics_f64_512", "kind": "uniform", "eq": "acoustics", "prec": "f64", "field": "const",
         "n": 32, "px": 16, "py": 16, "a": 0.0, "b": 0.0, "tune": True},
        # the benchmark's headline: 4096 x 4096 cells, state far larger than the cache
        {"name": "acoustics_f32_4096", "kind": "uniform", "eq": "acoustics", "prec": "f32", "field": "const",
         "n": 32, "px": 128, "py": 128, "a": 0.0, "b": 0.0, "tune": True},
        # swirl (the variable velocity of Section 4.3) on the benchmark's 4096 x 4096 cells in 16 x 16 patches
        {"name": "swirl_f32_4096", "kind": "uniform", "eq": "advection", "prec": "f32", "field": "swirl",
         "n": 16, "px": 256, "py": 256, "a": 0.0, "b": 0.0, "tune": False},
        # the state in pinned host memory, copied in and out by bands around every step
        {"name": "host_acoustics_f32_2048", "kind": "host", "eq": "acoustics", "prec": "f32", "field": "const",
         "n": 32, "px": 64, "py": 64, "a": 0.0, "b": 0.0, "tune": False, "bands": 32},
        # one subcycled coarse step of the adaptive ring wave, levels 3-7 on the 3 x 3 brick (configuration 4),
        # replayed from a graph
        {"name": "amr_acoustics_f32", "kind": "amr", "eq": "acoustics", "prec": "f32", "B": 3, "lmin": 3, "lmax": 7,
         "n": 16, "r0": 0.25, "w": 0.064, "copies": False, "a": 0.0, "b": 0.0},
        # adaptive advection of a wave packet per tree, levels 2-6 on the 2 x 2 brick, FP64 (configuration 3)
        {"name": "amr_advection_f64", "kind": "amr", "eq": "advection", "prec": "f64", "B": 2, "lmin": 2, "lmax": 6,
         "n": 16, "r0": 0.0, "w": 0.18, "copies": True, "a": 1.0, "b": 1.0},
        # the adaptive cycle with a changing forest: learned tags, regrid, coarse step, and back
        {"name": "regrid_acoustics_f32", "kind": "regrid", "eq": "acoustics", "prec": "f32", "B": 3, "lmin": 3,
         "lmax": 6, "n": 16, "r0": 0.25, "w": 0.064, "copies": False, "a": 0.0, "b": 0.0},
        # the learned tagger over a large forest's leaves (the benchmark's 65,536 patches)
        {"name": "tagger_infer_65536", "kind": "infer", "ncomp": 3, "n": 16, "batch": 65536},
        # one training step of the tagger on its default batch
        {"name": "tagger_train_4096", "kind": "train", "ncomp": 3, "n": 16, "batch": 4096},
    ]


def _log(rng, lo, hi):
    return lo * (hi / lo) ** rng.random()


def draw(rng):
    kind = rng.choice(("uniform", "uniform", "uniform", "host", "amr", "amr", "regrid", "infer", "train"))
    if kind in ("infer", "train"):
        n = rng.choice((8, 16, 16))
        top = 65536 if kind == "infer" else 8192
        return {"kind": kind, "ncomp": rng.choice((1, 3)), "n": n, "batch": int(_log(rng, 64, top))}
    eq = rng.choice(("advection", "acoustics"))
    prec = rng.choice(("f32", "f32", "f64"))
    a, b = ((round(rng.uniform(-1, 1), 3), round(rng.uniform(-1, 1), 3)) if eq == "advection" else (0.0, 0.0))
    if kind in ("amr", "regrid"):
        eq, prec = (eq, prec) if kind == "amr" else ("acoustics", "f32")
        case = {"kind": kind, "eq": eq, "prec": prec, "B": rng.choice((1, 2, 3)), "lmin": rng.choice((2, 3)), "lmax": 0,
                "n": rng.choice((8, 16, 16)) if kind == "amr" else 16,
                "r0": round(rng.choice((0.0, rng.uniform(0.15, 0.35))), 3), "w": round(rng.uniform(0.03, 0.12), 3),
                "copies": rng.random() < 0.5, "a": a if eq == "advection" else 0.0,
                "b": b if eq == "advection" else 0.0}
        # the finest level: one to four above the coarsest, as far as the cell updates of a coarse step allow
        area = math.pi * ((case["r0"] + case["w"]) ** 2 - max(0.0, case["r0"] - case["w"]) ** 2)
        area *= case["B"] ** 2 if case["copies"] else 1
        most = (1e6 if prec == "f64" and eq == "acoustics" else 12e6 if kind == "amr" else 4e6)
        fits = [m for m in (1, 2, 3, 4) if area * 4 ** (case["lmin"] + m) * 2 ** m * case["n"] ** 2 <= most] or [1]
        case["lmax"] = case["lmin"] + rng.choice(fits[-2:])
        return case
    if kind == "host":
        eq, a, b = "acoustics", 0.0, 0.0
    field = rng.choice(("const", "solid", "swirl")) if eq == "advection" and kind == "uniform" else "const"
    if field != "const":
        a = b = 0.0
    n = rng.choice((8, 16, 32, rng.randint(5, 64)))
    most = 16e6 if prec == "f32" and kind == "uniform" else 1e6 if prec == "f64" and field != "const" else 4e6
    cells = _log(rng, 64 * 64, most)
    px = max(1, round(math.sqrt(cells) / n * rng.uniform(0.7, 1.4)))
    py = max(1, round(cells / (n * n * px)))
    if field != "const" and px != py:
        py = px
    case = {"kind": kind, "eq": eq, "prec": prec, "field": field, "n": n, "px": px, "py": py, "a": a, "b": b,
            "tune": kind == "uniform" and field == "const" and rng.random() < 0.5}
    if kind == "host":
        case["bands"] = rng.choice((4, 16, 32))
    return case


# ------------------------------------------------------------------ initial data
def _wave(rng, count=4, top=6):
    """A smooth periodic function on the unit square, as [(amplitude, kx, ky, phase)]."""
    return [(rng.uniform(0.2, 1.0) / count, rng.randint(-top, top), rng.randint(-top, top),
             rng.uniform(0, 2 * math.pi)) for _ in range(count)]


def _data(case, seed):
    """Callables f(x, y), one per component, periodic on the case's domain: long waves, and what the workload
    is about on top (a pulse and a vortex, a ring wave, a packet)."""
    rng = random.Random(seed)
    ncomp = 3 if case["eq"] == "acoustics" else 1
    adaptive, r0 = "lmax" in case, case.get("r0", 0.0)
    amp, ph = rng.uniform(0.5, 1.5), rng.uniform(0, 2 * math.pi)
    cx, cy = rng.uniform(0.4, 0.6), rng.uniform(0.4, 0.6)
    modes = [_wave(rng) for _ in range(ncomp)]

    def component(c):
        def f(x, y):
            if not adaptive:
                v = 0.0
                # the rotating box does not wrap around: its data vanish near the edges
                for a, kx, ky, p in modes[c] if case["field"] != "solid" else ():
                    v = v + a * torch.sin(2 * math.pi * (kx * x + ky * y) + p)
                px, py = torch.remainder(x, 1.0) - cx, torch.remainder(y, 1.0) - cy
                pulse = amp * torch.exp(-(px * px + py * py) / 0.005)
                return v + (pulse if c == 0 else (-py if c == 1 else px) * 5.0 * pulse)
            if c > 0:
                return 0.0 * x + 0.0 * y
            px, py = _folded(case, x), _folded(case, y)
            r = torch.sqrt(px * px + py * py)
            if r0 > 0:
                return amp * torch.exp(-((r - r0) ** 2) / 0.001) * torch.cos(80 * math.pi * r + ph)
            return amp * torch.exp(-r * r / 0.01) * torch.cos(60 * math.pi * px + ph)
        return f
    return [component(c) for c in range(ncomp)]


def _folded(case, x):
    """Coordinate relative to the centre the data is placed on: the domain's, or every unit tree's."""
    if case["copies"]:
        return (torch.remainder(x, 1.0) if torch.is_tensor(x) else np.mod(x, 1.0)) - 0.5
    B = case["B"]
    return (torch.remainder(x, B) if torch.is_tensor(x) else np.mod(x, B)) - 0.5 * B


def _planes(f, xl, yl, dx, dy):
    """The four planes of one component on lattice lines xl, yl (last axis x): cell averages by 2 x 2 Gauss
    points, left-edge, corner and bottom-edge values."""
    g = 0.5 / math.sqrt(3.0)
    X, Y = xl[..., None, :], yl[..., :, None]
    dX, dY = dx[..., None, None], dy[..., None, None]
    avg = 0.0
    for sx in (-g, g):
        for sy in (-g, g):
            avg = avg + 0.25 * f(X + (0.5 + sx) * dX, Y + (0.5 + sy) * dY)
    return [avg, f(X, Y + 0.5 * dY), f(X, Y), f(X + 0.5 * dX, Y)]


def _fill_uniform(state, case, seed, lo, dx, dy):
    """Initial values of a uniform run's state [patches, words] on the GPU, ghost rings included."""
    n, px, py, dev = case["n"], case["px"], case["py"], state.device
    W = n + 2 * G + 1
    ncomp = 3 if case["eq"] == "acoustics" else 1
    st = state.view(px * py, ncomp, 4, -1)
    st[..., W * W:] = 0
    xl = lo[0] + torch.arange(-G, px * n + G + 1, device=dev, dtype=torch.float64) * dx
    yl = lo[1] + torch.arange(-G, py * n + G + 1, device=dev, dtype=torch.float64) * dy
    one = torch.ones((), device=dev, dtype=torch.float64)
    for c, f in enumerate(_data(case, seed)):
        h = lambda x, y, f=f: f((x - lo[0]) / (px * n * dx), (y - lo[1]) / (py * n * dy))  # noqa: E731
        for k, plane in enumerate(_planes(h, xl, yl, dx * one, dy * one)):
            st[:, c, k, :W * W] = plane.unfold(0, W, n).unfold(1, W, n).reshape(px * py, W * W).to(state.dtype)


def _owned(state, n, ncomp):
    """View of the degrees of freedom the patches own: [patches, ncomp, 4, n, n]."""
    W = n + 2 * G + 1
    st = state.view(state.shape[0], ncomp, 4, -1)[..., :W * W].unflatten(-1, (W, W))
    return st[..., G:G + n, G:G + n]


# --------------------------------------------------------------------- preparing
def _geometry(case):
    """Lower-left corner, mesh widths and time step of a uniform case."""
    n, px, py = case["n"], case["px"], case["py"]
    lo, size = ((-1.0, -1.0), 2.0) if case["field"] == "solid" else ((0.0, 0.0), 1.0)
    dx, dy = size / (px * n), size / (py * n)
    if case["field"] == "solid":
        dt = 0.45 * min(dx, dy) / (math.pi * (1.0 + 3 * max(dx, dy)))
    elif case["field"] == "swirl":
        dt = 0.45 * min(dx, dy)
    elif case["eq"] == "advection":
        dt = CFL / max(abs(case["a"]) / dx, abs(case["b"]) / dy, 1e-3 / dx)
    else:
        dt = CFL * min(dx, dy)
    return lo, dx, dy, dt


def _config(case):
    eq = af.ACOUSTICS if case["eq"] == "acoustics" else af.ADVECTION
    return af.config(eq, PREC[case["prec"]], case["n"], case["a"], case["b"], 1.0)


def _key(case):
    return tuple(sorted((k, str(v)) for k, v in case.items() if k != "name"))


def _prepare_uniform(case, seed):
    lo, dx, dy, dt = _geometry(case)
    t0 = 0.125 if case["field"] == "swirl" else 0.0
    run = UniformRun(_config(case), case["px"], case["py"], dx, dy, dt, field=FIELD[case["field"]], lo=lo, t0=t0)
    if case["tune"]:
        # the package's autotuner, as the benchmark uses it: once per workload and process
        _fill_uniform(run.state, case, seed, lo, dx, dy)
        tune.tune(run, key=_key(case))
        run.t = t0
    _fill_uniform(run.a, case, seed, lo, dx, dy)
    run.b.copy_(run.a)
    # what a program looks at after a step: views of the two buffers, made once
    state = {"case": case, "run": run, "first": run.a,
             "views": [_owned(buf, case["n"], run.cfg.ncomp) for buf in (run.a, run.b)]}
    if case["kind"] == "host":
        own = _owned(run.a, case["n"], 3).reshape(run.npatch, -1)
        host = torch.empty(own.shape, dtype=own.dtype, pin_memory=True)
        host.copy_(own)
        state["host"] = host
    return state


def _adapted(case):
    """Leaves (level, ix, iy) of the case's forest: from the coarsest level, every patch that meets the band
    |r - r0| <= w is refined until lmax, by the package's own regrid rule (2:1 balanced)."""
    B, lmin, lmax = case["B"], case["lmin"], case["lmax"]
    side = B << lmin
    iy, ix = (v.reshape(-1).astype(np.int32) for v in np.mgrid[0:side, 0:side])
    arrays = (np.full(side * side, lmin, np.int32), ix, iy)
    for _ in range(lmax - lmin):
        F = Forest(B, lmax, device="cpu", arrays=arrays)
        w = 1.0 / (1 << F.level)
        near, far = [], []
        for i in (F.ix, F.iy):
            mid, half = _folded(case, (i + 0.5) * w), 0.5 * w
            near.append(np.maximum(np.abs(mid) - half, 0.0))
            far.append(np.abs(mid) + half)
        meets = (np.hypot(*near) <= case["r0"] + case["w"]) & (np.hypot(*far) >= case["r0"] - case["w"])
        arrays = regrid_arrays(F, np.where(meets & (F.level < lmax), 1, 0).astype(np.int8), lmin)
    return Forest(B, lmax, device="cpu", arrays=arrays)


class _Coarse:
    """An adaptive run as the autotuner takes it."""

    def __init__(self, run):
        self.set_tiling, self.step = run.set_tiling, run.coarse_step


def _fill_forest(run, case, seed):
    F, n, dev = run.forest, case["n"], run.a.device
    W, ncomp = n + 2 * G + 1, run.cfg.ncomp
    lev, ix, iy = (torch.from_numpy(v.astype(np.float64)).to(dev) for v in (F.level, F.ix, F.iy))
    w = 1.0 / 2.0 ** lev
    d = w / n
    k = torch.arange(-G, n + G + 1, device=dev, dtype=torch.float64)
    xl, yl = (ix * w)[:, None] + k * d[:, None], (iy * w)[:, None] + k * d[:, None]
    st = run.a.view(F.nleaf, ncomp, 4, -1)
    for c, f in enumerate(_data(case, seed)):
        for q, plane in enumerate(_planes(f, xl, yl, d, d)):
            st[:, c, q, :W * W] = plane.reshape(F.nleaf, W * W).to(run.a.dtype)


def _prepare_amr(case, seed):
    F = _adapted(case)
    cfg = _config(case)
    leaves = F.leaves
    speed = max(abs(case["a"]), abs(case["b"]), 1e-3) if case["eq"] == "advection" else 1.0
    dt0 = CFL / case["n"] / speed
    zero = np.zeros((len(leaves), af.patch_words(cfg.n, cfg.ncomp)), np.float32 if case["prec"] == "f32" else np.float64)
    run = AMRRun(cfg, case["B"], case["lmax"], leaves, zero, (0.0, 0.0), (float(case["B"]),) * 2, dt0)
    tune.tune(_Coarse(run), key=_key(case), steps=3, warmup=1)  # without graphs: each would be captured anew
    run.use_graphs = case["kind"] == "amr"
    for buf in (run.a, run.b, run.freg):  # the tuner's own steps are forgotten
        buf.zero_()
    run.parity, run.time = 0, 0.0
    _fill_forest(run, case, seed)
    run.fill(run.all_levels, run.all_levels)
    state = {"case": case, "run": run, "views": _leaf_views(run)}
    if case["kind"] == "regrid":
        # half of the leaves that can be split and merged again without a cascade: those among equals, whose
        # parent's neighbours are all refined
        rng = np.random.default_rng(0)
        free = [l < case["lmax"] and (l == case["lmin"] or all(
            F.region(l - 1, (x >> 1) + i, (y >> 1) + j) < 0 for i in (-1, 0, 1) for j in (-1, 0, 1)))
            for l, x, y in leaves]
        up = ((F.nbr >= 0).all(axis=1) & np.array(free) & (rng.random(F.nleaf) < 0.5)).astype(np.int8)
        N = Forest(F.B, F.lmax, device="cpu", arrays=regrid_arrays(F, up, case["lmin"]))
        split = {(l + 1, x, y) for l, x, y in (t for t, u in zip(leaves, up) if u)}
        down = np.array([-1 if (l, x >> 1, y >> 1) in split else 0 for l, x, y in N.leaves], np.int8)
        state |= {"up": up, "down": down, "tagger": Tagger(cfg.ncomp, cfg.n, seed=seed % 5)}
    return state


def _samples(case, seed):
    """Tagger inputs: patches of plane waves of all lengths and strengths around the tagging threshold, labelled
    by the central difference of the first component."""
    ns, C, S = case["batch"], case["ncomp"], case["n"] + 4
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.rand((5, ns, C, 1, 1), generator=g, device="cuda")
    y, x = torch.meshgrid(*(torch.arange(S, device="cuda", dtype=torch.float32),) * 2, indexing="ij")
    amp, k, th, ph = torch.exp(8 * u[0] - 4), 0.1 + 1.4 * u[1], 6.2832 * u[2], 6.2832 * u[3]
    v = amp * torch.sin(k * (torch.cos(th) * x + torch.sin(th) * y) + ph)
    v = v - v[..., 2:-2, 2:-2].mean(dim=(-1, -2), keepdim=True)
    p = v[:, 0]
    d = torch.maximum((p[:, 3:-3, 4:-2] - p[:, 3:-3, 2:-4]).abs().amax((1, 2)),
                      (p[:, 4:-2, 3:-3] - p[:, 2:-4, 3:-3]).abs().amax((1, 2)))
    label = (d >= 1.0).float()
    level = torch.randint(2, 8, (ns,), generator=g, device="cuda", dtype=torch.int32)
    return v.to(torch.bfloat16).contiguous().view(torch.int16), level, label


def _prepare_tagger(case, seed):
    x, level, label = _samples(case, seed)
    tg = Tagger(case["ncomp"], case["n"], seed=seed % 1000)
    weight = torch.where(label > 0.5, 1.0, 0.6)
    return {"case": case, "tagger": tg, "x": x, "level": level, "label": label, "weight": weight,
            "wsum": float(weight.sum().item()), "out": tg.outputs(case["batch"])}


def prepare(case, seed):
    if case["kind"] in ("uniform", "host"):
        return _prepare_uniform(case, seed)
    if case["kind"] in ("amr", "regrid"):
        return _prepare_amr(case, seed)
    return _prepare_tagger(case, seed)


# ----------------------------------------------------------------------- running
def _leaf_views(run):
    """The owned degrees of freedom of every level, in both buffers."""
    return {l: [_owned(buf[run.forest.level_slice(l)], run.cfg.n, run.cfg.ncomp) for buf in (run.a, run.b)]
            for l in run.forest.levels}


def _current(run, views):
    """Of every level the view of the buffer that holds its current values."""
    return {f"level{l}": v[(run.parity >> l) & 1] for l, v in views.items()}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "uniform":
        r = state["run"]
        r.step()
        return state["views"][r.state is not state["first"]]
    if kind == "host":
        state["run"].step_host_owned(state["host"], case["bands"])
        return state["host"]
    if kind == "amr":
        r = state["run"]
        r.coarse_step()
        return _current(r, state["views"])
    if kind == "regrid":
        r = state["run"]
        tags, nfall = r.tags_learned(state["tagger"], 0, 1, 4.0, 1.0, 0.1)
        r.regrid(state["up"], case["lmin"])
        r.coarse_step()
        r.regrid(state["down"], case["lmin"])
        r.coarse_step()
        return {"tags": tags, "fallbacks": nfall, "level": r.forest.level, **_current(r, _leaf_views(r))}
    tg = state["tagger"]
    if kind == "infer":
        logit, m = tg.infer(state["x"], state["level"], state["out"][:2])
        return {"logit": logit, "maxima": m}
    logit, m, arg = tg.train_step(state["x"], state["level"], state["label"], state["weight"], state["wsum"], 1e-4,
                                  state["out"])
    return {"logit": logit, "maxima": m, "positions": arg, "grad": tg.grad, "params": tg.params, "m": tg.m, "v": tg.v}


# -------------------------------------------------------------------------- work
def work(case):
    kind = case["kind"]
    if kind in ("infer", "train"):
        ns, C, n = case["batch"], case["ncomp"], case["n"]
        nparam = 32 * C * 9 + 16 * 32 + 32 * 32 * 9 + 32 + 32 + 1
        fwd = 2 * 32 * ((n + 2) ** 2 * C * 9 + n * n * 32 * 9)
        b = ns * (2 * C * (n + 4) ** 2 + 4 + 4 + 4 * 32) + 4 * nparam
        if kind == "infer":
            return {"bytes": b, "flops": ns * fwd}
        # one pixel per channel carries the gradient back: 9 x 32 taps to the weights of the second layer and
        # to its inputs, and from at most 288 pixels of the first layer's map to the weights of the first
        back = 2 * 2 * 32 * 9 * 32 + 2 * 288 * 32 * C * 9 // 4
        return {"bytes": b + ns * (4 * 32 + 8) + 7 * 4 * nparam, "flops": ns * (fwd + back)}
    size = 4 if case["prec"] == "f32" else 8
    ncomp = 3 if case["eq"] == "acoustics" else 1
    # acoustics: the folded stencils of three nodes and the fluxes; advection: two evaluations of the
    # reconstruction at three nodes and the fluxes; variable velocity: feet by one Runge-Kutta step (eight
    # velocities) or a rotation each besides
    per_cell = 750 if ncomp == 3 else 3 * 2 * 17 + 28
    if case.get("field", "const") != "const":
        per_cell = 3 * 2 * (60 + (4 * 40 if case["field"] == "swirl" else 10)) + 80
    if kind in ("uniform", "host"):
        cells = case["px"] * case["py"] * case["n"] ** 2
        return {"bytes": 2 * 4 * ncomp * size * cells, "flops": per_cell * cells}
    F = _adapted(case)
    lo = int(F.level.min())
    cells = int(((1 << (F.level - lo)).astype(np.int64) * case["n"] ** 2).sum())
    w = {"bytes": 2 * 4 * ncomp * size * cells, "flops": per_cell * cells}
    if kind == "regrid":  # two coarse steps, and the state moved twice to another forest
        w = {k: 2 * v for k, v in w.items()}
        w["bytes"] += 2 * 2 * 4 * ncomp * size * F.nleaf * case["n"] ** 2
    return w


# ------------------------------------------------------------------------- exact
def _global(own, px, py, n):
    """[patches, ncomp, 4, n, n] as global periodic arrays [ncomp][4] of [py n, px n], in 64 bits."""
    o = own.double().view(py, px, -1, 4, n, n).permute(2, 3, 0, 4, 1, 5).reshape(-1, 4, py * n, px * n)
    return [[o[c, k] for k in range(4)] for c in range(o.shape[0])]


def _patches(q, px, py, n):
    o = torch.stack([torch.stack(c) for c in q])
    return o.view(-1, 4, py, n, px, n).permute(2, 4, 0, 1, 3, 5).reshape(px * py, -1, 4, n, n)


def _at(a, i, j):
    """Periodic array a shifted so that entry (y, x) is a[y + j, x + i]."""
    return torch.roll(a, (-j, -i), (0, 1)) if i or j else a


def _nodal(planes, i, j):
    """The 3 x 3 nodal values (row by row) of the reconstruction of cell (x + i, y + j)."""
    avg, xm, co, ym = planes
    c00, c10, c01, c11 = (_at(co, i + a, j + b) for b in (0, 1) for a in (0, 1))
    xl, xr, yb, yt = _at(xm, i, j), _at(xm, i + 1, j), _at(ym, i, j), _at(ym, i, j + 1)
    cen = 2.25 * _at(avg, i, j) - (c00 + c10 + c01 + c11) / 16 - (xl + xr + yb + yt) / 4
    return [c00, yb, c10, xl, cen, xr, c01, yt, c11]


def _lagrange(s):
    """Values and derivatives of the three quadratic Lagrange polynomials on {-1, 0, 1}."""
    return ([s * (s - 1) / 2, 1 - s * s, s * (s + 1) / 2], [s - 0.5, -2 * s, s + 0.5])


# node types: corner, left-edge midpoint, bottom-edge midpoint; for each the cells that its disc meets, as
# (cell offset, node in the cell's coordinates, angular sector)
_H = 0.5 * math.pi
_SECTORS = [
    [(0, 0, -1, -1, 0, _H), (-1, 0, 1, -1, _H, 2 * _H), (-1, -1, 1, 1, 2 * _H, 3 * _H), (0, -1, -1, 1, 3 * _H, 4 * _H)],
    [(0, 0, -1, 0, -_H, _H), (-1, 0, 1, 0, _H, 3 * _H)],
    [(0, 0, 0, -1, 0, 2 * _H), (0, -1, 0, 1, 2 * _H, 4 * _H)],
]


def _sphere_weights(xin, etan, p0, p1, R, dx, dy):
    """Nodal weights of M + R d_R M, -R M d/dx and -R M d/dy over one sector of the disc of radius R, by
    Gauss quadrature (the integrands are polynomials in the sine and cosine of both angles)."""
    g, w = np.polynomial.legendre.leggauss(24)
    th, wt = (g + 1) * _H / 2, w * _H / 2
    ph, wp = p0 + (g + 1) * (p1 - p0) / 2, w * (p1 - p0) / 2
    TH, PH = np.meshgrid(th, ph)
    W = np.outer(wp, wt) * np.sin(TH) / (2 * math.pi)
    X, Y = R * np.sin(TH) * np.cos(PH), R * np.sin(TH) * np.sin(PH)
    lx, dlx = _lagrange(xin + 2 * X / dx)
    ly, dly = _lagrange(etan + 2 * Y / dy)
    out = []
    for b in range(3):
        for a in range(3):
            fx, fy = dlx[a] * ly[b] * 2 / dx, lx[a] * dly[b] * 2 / dy
            out.append([float((W * v).sum()) for v in (lx[a] * ly[b] + X * fx + Y * fy, -R * fx, -R * fy)])
    return out


def _acoustic_nodes(q, tau, dx, dy):
    """Point values of the three node types after tau, [type][comp] (c = 1)."""
    out = [[0.0] * 3 for _ in range(3)]
    for t, sectors in enumerate(_SECTORS):
        for i, j, xin, etan, p0, p1 in sectors:
            w = _sphere_weights(xin, etan, p0, p1, tau, dx, dy)
            p, u, v = (_nodal(c, i, j) for c in q)
            for k, (m, wx, wy) in enumerate(w):
                out[t][0] = out[t][0] + m * p[k] + wx * u[k] + wy * v[k]
                out[t][1] = out[t][1] + m * u[k] + wx * p[k]
                out[t][2] = out[t][2] + m * v[k] + wy * p[k]
    return out


def _value_at(planes, fx, fy):
    """The reconstruction at (fx, fy) (tensors, in cells from the domain's corner)."""
    ny, nx = fx.shape
    ci, cj = torch.floor(fx), torch.floor(fy)
    lx, ly = _lagrange(2 * (fx - ci) - 1)[0], _lagrange(2 * (fy - cj) - 1)[0]
    ci, cj = torch.remainder(ci, nx).long(), torch.remainder(cj, ny).long()
    q = _nodal(planes, 0, 0)
    return sum(lx[a] * ly[b] * q[3 * b + a][cj, ci] for b in range(3) for a in range(3))


def _foot(case, x, y, t, tau, dx, dy):
    if case["field"] == "solid":
        c, s = math.cos(math.pi * tau), math.sin(math.pi * tau)
        return x * c + y * s, -x * s + y * c
    k1 = _swirl(x, y, t + tau, dx, dy)
    k2 = _swirl(x - tau / 2 * k1[0], y - tau / 2 * k1[1], t + tau / 2, dx, dy)
    k3 = _swirl(x - tau / 2 * k2[0], y - tau / 2 * k2[1], t + tau / 2, dx, dy)
    k4 = _swirl(x - tau * k3[0], y - tau * k3[1], t, dx, dy)
    return tuple(z - tau / 6 * (k1[i] + 2 * k2[i] + 2 * k3[i] + k4[i]) for i, z in enumerate((x, y)))


def _swirl(x, y, t, dx, dy):
    """Centred differences over one mesh width of sin^2(pi x) sin^2(pi y) cos(pi t) / pi."""
    psi = lambda a, b: (torch.sin(math.pi * a) * torch.sin(math.pi * b)) ** 2 * math.cos(math.pi * t) / math.pi  # noqa: E731
    return (-(psi(x, y + dy / 2) - psi(x, y - dy / 2)) / dy, (psi(x + dx / 2, y) - psi(x - dx / 2, y)) / dx)


def _exact_step(case, q, dx, dy, dt, lo, t0):
    """One Active Flux step of global periodic arrays q[comp][plane]."""
    ny, nx = q[0][0].shape
    dev = q[0][0].device
    times = [[[c[k] for c in q] for k in (2, 1, 3)]]  # [time][type][comp]
    X = lo[0] + torch.arange(nx, device=dev, dtype=torch.float64)[None, :] * dx + torch.zeros((ny, 1), device=dev)
    Y = lo[1] + torch.arange(ny, device=dev, dtype=torch.float64)[:, None] * dy + torch.zeros((1, nx), device=dev)
    for tau in (dt / 2, dt):
        if len(q) == 3:
            times.append(_acoustic_nodes(q, tau, dx, dy))
            continue
        nodes = []
        for ox, oy in ((0.0, 0.0), (0.0, 0.5), (0.5, 0.0)):
            x, y = X + ox * dx, Y + oy * dy
            if case["field"] == "const":
                i, j = torch.round((X - lo[0]) / dx), torch.round((Y - lo[1]) / dy)
                fx, fy = i + (ox - case["a"] * tau / dx), j + (oy - case["b"] * tau / dy)
            else:
                xf, yf = _foot(case, x, y, t0, tau, dx, dy)
                fx, fy = (xf - lo[0]) / dx, (yf - lo[1]) / dy
            nodes.append([_value_at(q[0], fx, fy)])
        times.append(nodes)
    new = []
    for c in range(len(q)):
        F = Gy = 0.0  # 36 times the fluxes through the left and bottom faces
        for k, (w, nodes) in enumerate(zip((1, 4, 1), times)):
            a = b = 1.0
            f = g = c  # the component whose values the flux takes: acoustics f = (u, p, 0), g = (v, 0, p)
            if len(q) == 3:
                f, g = (1, 0, None)[c], (2, None, 0)[c]
            elif case["field"] == "const":
                a, b = case["a"], case["b"]
            elif case["field"] == "swirl":
                a = _swirl(X, Y + dy / 2, t0 + k * dt / 2, dx, dy)[0]
                b = _swirl(X + dx / 2, Y, t0 + k * dt / 2, dx, dy)[1]
            va = [-math.pi * (Y + o * dy) if case["field"] == "solid" else a for o in (0, 0.5, 1)]
            vb = [math.pi * (X + o * dx) if case["field"] == "solid" else b for o in (0, 0.5, 1)]
            if f is not None:
                pts = (nodes[0][f], nodes[1][f], _at(nodes[0][f], 0, 1))
                F = F + w * sum(s * v * z for s, v, z in zip((1, 4, 1), va, pts))
            if g is not None:
                pts = (nodes[0][g], nodes[2][g], _at(nodes[0][g], 1, 0))
                Gy = Gy + w * sum(s * v * z for s, v, z in zip((1, 4, 1), vb, pts))
        avg = q[c][0]
        if torch.is_tensor(F):
            avg = avg - dt / dx / 36 * (_at(F, 1, 0) - F)
        if torch.is_tensor(Gy):
            avg = avg - dt / dy / 36 * (_at(Gy, 0, 1) - Gy)
        n = times[2]
        new.append([avg, n[1][c], n[0][c], n[2][c]])
    return new


def _bf16(v):
    return v.to(torch.bfloat16).double()


def _exact_tagger(case, seed):
    """The network in 64 bits on the stored values: inputs, convolution weights and the first map are BF16."""
    x, level, label = _samples(case, seed)
    C, ns = case["ncomp"], case["batch"]
    p0 = Tagger(C, case["n"], seed=seed % 1000).params.double()
    p = p0.clone().requires_grad_(case["kind"] == "train")
    sizes = [32 * C * 9, 16 * 32, 32 * 32 * 9, 32, 32, 1]

    class Round(torch.autograd.Function):  # BF16 storage; its gradient passes unchanged
        @staticmethod
        def forward(ctx, v):
            return _bf16(v)

        @staticmethod
        def backward(ctx, g):
            return g

    logits, maxima, places, grad = [], [], [], torch.zeros_like(p0)
    weight = torch.where(label > 0.5, 1.0, 0.6).double()
    for s in range(0, ns, 4096):
        e = min(ns, s + 4096)
        w1, emb, w2, b2, w3, b3 = p.split(sizes)
        w1, w2 = Round.apply(w1).view(32, C, 3, 3), Round.apply(w2).view(32, 32, 3, 3)
        xs = x[s:e].view(torch.bfloat16).double()
        conv = lambda a, w: torch.nn.functional.conv2d(a, w)  # noqa: E731
        z = Round.apply(torch.relu(conv(xs, w1) + emb.view(16, 32)[level[s:e].long()][:, :, None, None]))
        z = (conv(z, w2) + b2[None, :, None, None]).flatten(2)
        top, at = z.max(dim=2)
        m = torch.relu(top)
        logit = m @ w3 + b3
        if case["kind"] == "train":
            y, om = label[s:e].double(), weight[s:e]
            loss = (om * torch.nn.functional.binary_cross_entropy_with_logits(logit, y, reduction="none")).sum()
            grad += torch.autograd.grad(loss, p)[0]
        logits.append(logit.detach())
        maxima.append(m.detach())
        places.append(torch.where(top.detach() > 0, at, -1))
    logit, m = torch.cat(logits), torch.cat(maxima)
    if case["kind"] == "infer":
        return {"logit": logit, "maxima": m}
    grad /= float(weight.sum().item())
    return {"logit": logit, "maxima": m, "positions": None, "grad": grad, "params": None, "m": 0.1 * grad,
            "v": 0.001 * grad * grad}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("infer", "train"):
        return _exact_tagger(case, seed)
    if kind not in ("uniform", "host"):
        return None  # an adaptive coarse step has no short plain restatement
    n, px, py = case["n"], case["px"], case["py"]
    lo, dx, dy, dt = _geometry(case)
    ncomp = 3 if case["eq"] == "acoustics" else 1
    dtype = torch.float32 if case["prec"] == "f32" else torch.float64
    st = torch.zeros((px * py, af.patch_words(n, ncomp)), dtype=dtype, device="cuda")
    _fill_uniform(st, case, seed, lo, dx, dy)
    q = _global(_owned(st, n, ncomp), px, py, n)
    t0 = 0.125 if case["field"] == "swirl" else 0.0
    new = _patches(_exact_step(case, q, dx, dy, dt, lo, t0), px, py, n)
    return new.reshape(px * py, -1) if kind == "host" else new
