"""The work that users of this framework have it do, as cases that can be timed.

A case is a plain dict; `prepare` makes its inputs and the handles a program
keeps (stencils, contexts, networks), `run` is one pass through the public
entry points and returns what the pass computes, `work` counts the bytes and
operations that a pass cannot do without, and `exact` gives the same outputs
from plain torch arithmetic in 64 bits.

Node sets are the repository's own seeded generators.  A node set and its
stencils belong to the case (a program builds them once and runs many flows
on them), so they are kept per process; the flow's initial state, network or
device arrays come from the seed.  The solver's state is FP32; its getters
widen it to float64, and the programs here keep it in the state's own
precision, as FP32 tensors.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2312_14789_gb300 import inputs as I
from paper_2312_14789_gb300 import mlbm as M
from paper_2312_14789_gb300 import warmstart

U0 = 0.05  # maximum inflow velocity of the vortex street
LAMBDA = 3.0 / 16.0  # (tau+ - 1/2)(tau- - 1/2) of the TRT runs


def listed():
    return [
        # The plain-MLBM Poiseuille channel (2000 nodes): the smallest run, bound by the time per launch.
        {"name": "channel_2k", "kind": "channel", "nx": 40, "ny": 50, "geo": 1, "K": 12, "s": 1.0, "bb": 1,
         "model": "bgk", "tau": 0.8, "trt": False, "g": 1e-6, "steps": 200},
        # One porous sample (the warm-start configuration, ~192k nodes, Darcy flow) on its way to the steady
        # state: the criterion every 100 steps, then the observables and the fields.
        {"name": "porous_steady", "kind": "steady", "n": 200_000, "phi": 0.7, "geo": 20_000, "s": 1.0, "g": 1e-6,
         "window": 200, "check": 100, "steps": 400},
        # Many flows through one sample in one batched context (streaming distances 1, 1/2, 1/4 and body
        # forces from Darcy to inertial): larger than the L2, the framework's headline workload in kind.
        {"name": "porous_batch", "kind": "batch", "n": 200_000, "phi": 0.7, "geo": 20_000, "runs": 9,
         "steps": 128},
        # The two-relaxation-time BGK state on a porous sample with interpolated bounce-back.
        {"name": "porous_trt", "kind": "porous", "n": 100_000, "phi": 0.7, "geo": 10_000, "K": 16, "s": 0.5,
         "bb": 1, "model": "bgk", "tau": 0.8, "trt": True, "g": 1e-6, "steps": 100},
        # The vortex street behind a cylinder on the scattered node set (~260k nodes), forces every 50 steps.
        {"name": "vortex", "kind": "vortex", "scale": 1.0, "geo": 2, "hybrid": False, "s": 0.5, "re": 100.0,
         "interp": "wls", "every": 50, "records": 4},
        # The same flow on the hybrid set: regular lattice with scattered refinement (~165k nodes).
        {"name": "vortex_hybrid", "kind": "vortex", "scale": 1.0, "geo": 2, "hybrid": True, "s": 0.5, "re": 100.0,
         "interp": "wls", "every": 50, "records": 4},
        # The paper's RBF-FD interpolant, a stencil per Lagrangian point, on a smaller vortex street.
        {"name": "vortex_rbf", "kind": "vortex", "scale": 0.5, "geo": 2, "hybrid": False, "s": 0.5, "re": 100.0,
         "interp": "points", "every": 50, "records": 2},
        # The lattice LBM that the paper compares with (D = 80 spacings), forces every 50 steps.
        {"name": "lattice_80", "kind": "lattice", "d": 80, "re": 100.0, "every": 50, "records": 20},
        # One node set split into four ranges, with the halo exchange of every step.
        {"name": "partition_4", "kind": "part", "n": 100_000, "phi": 0.7, "geo": 10_000, "s": 1.0, "g": 1e-6,
         "parts": 4, "steps": 100},
        # Training the warm-start network: Adam on minibatches drawn from a large training set.
        {"name": "net_train", "kind": "train", "rows": 1_000_003, "batch": 65_536, "outs": 3, "lr": 1e-3,
         "steps": 16},
        # Starting a new sample from the network: features of its nodes, prediction, initial state.
        {"name": "warm_start", "kind": "warm", "n": 200_000, "phi": 0.7, "geo": 20_000, "outs": 3, "g": 1e-6},
        # The area-weighted sums of a caller's own device arrays (all samples of a large study).
        {"name": "sums_device", "kind": "sums", "n": 13_254_482, "mask": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["channel", "channel", "porous", "steady", "batch", "vortex", "vortex", "lattice", "part",
                       "train", "warm", "sums"])
    geo = rng.randrange(1, 1_000_000)
    phi = round(rng.uniform(0.55, 0.85), 3)
    g = rng.choice([1e-6, 5e-6, 2e-5])
    if kind == "channel":
        tau1 = rng.random() < 0.4
        return {"kind": kind, "nx": _log_int(rng, 20, 500), "ny": _log_int(rng, 20, 400), "geo": geo,
                "K": rng.choice([12, 16, 24]), "s": rng.choice([0.5, 1.0]), "bb": rng.choice([0, 1]),
                "model": "tau1" if tau1 else "bgk", "tau": 1.0 if tau1 else round(rng.uniform(0.65, 1.1), 3),
                "trt": (not tau1) and rng.random() < 0.5, "g": 1e-6, "steps": rng.randrange(20, 200)}
    if kind == "porous":
        return {"kind": kind, "n": _log_int(rng, 5_000, 60_000), "phi": phi, "geo": geo, "K": 16,
                "s": rng.choice([0.5, 0.25]), "bb": rng.choice([0, 1]), "model": "bgk",
                "tau": round(rng.uniform(0.7, 1.0), 3), "trt": rng.random() < 0.5, "g": 1e-6,
                "steps": rng.randrange(20, 150)}
    if kind == "steady":
        check = rng.choice([50, 100])
        return {"kind": kind, "n": _log_int(rng, 5_000, 60_000), "phi": phi, "geo": geo,
                "s": rng.choice([1.0, 0.5, 0.25]), "g": g, "window": check * rng.choice([1, 2, 4]), "check": check,
                "steps": check * rng.randrange(4, 8)}
    if kind == "batch":
        return {"kind": kind, "n": _log_int(rng, 5_000, 60_000), "phi": phi, "geo": geo,
                "runs": rng.randrange(2, 17), "steps": rng.randrange(20, 150)}
    if kind == "vortex":
        points = rng.random() < 0.4
        return {"kind": kind, "scale": round(rng.uniform(0.2, 0.4 if points else 0.6), 3), "geo": geo,
                "hybrid": (not points) and rng.random() < 0.5, "s": rng.choice([0.5, 0.25]),
                "re": rng.choice([50.0, 100.0]), "interp": "points" if points else rng.choice(["wls", "wls", "rbf"]),
                "every": rng.randrange(20, 60), "records": rng.randrange(1, 5)}
    if kind == "lattice":
        return {"kind": kind, "d": _log_int(rng, 12, 110), "re": rng.choice([20.0, 100.0]),
                "every": 2 * rng.randrange(10, 40), "records": rng.randrange(2, 12)}
    if kind == "part":
        return {"kind": kind, "n": _log_int(rng, 5_000, 60_000), "phi": phi, "geo": geo,
                "s": rng.choice([1.0, 0.5]), "g": g, "parts": rng.randrange(2, 9), "steps": rng.randrange(10, 100)}
    if kind == "train":
        rows = _log_int(rng, 20_000, 2_000_000)
        return {"kind": kind, "rows": rows, "batch": min(rows, _log_int(rng, 1_000, 65_536)),
                "outs": rng.choice([2, 3]), "lr": rng.choice([1e-3, 3e-4]), "steps": rng.randrange(1, 17)}
    if kind == "warm":
        return {"kind": kind, "n": _log_int(rng, 5_000, 60_000), "phi": phi, "geo": geo, "outs": rng.choice([2, 3]),
                "g": g}
    return {"kind": kind, "n": _log_int(rng, 1_000, 13_000_000), "mask": rng.random() < 0.5}


# ------------------------------------------------------------------ node sets
@functools.lru_cache(maxsize=16)
def _porous(n, phi, geo):
    return I.porous_from_spec({"seed": geo, "n_target": n, "porosity": phi})


@functools.lru_cache(maxsize=16)
def _vortex(scale, geo, hybrid):
    return I.karman(seed=geo, scale=scale, lattice_beyond_d=1.0 if hybrid else None, areas="spacing")


@functools.lru_cache(maxsize=16)
def _channel(nx, ny, geo):
    return I.poiseuille_channel(nx, ny, 0.2, seed=geo)


def _node_set(c):
    if c["kind"] == "channel":
        return _channel(c["nx"], c["ny"], c["geo"])
    if c["kind"] == "vortex":
        return _vortex(c["scale"], c["geo"], c["hybrid"])
    return _porous(c["n"], c["phi"], c["geo"])


def _rule(c):
    """Stencil arguments of a case: K, s, bounce-back rule and interpolant."""
    if c["kind"] == "vortex":
        K = {"wls": 16, "rbf": 24, "points": 64}[c["interp"]]
        interp = {"wls": M.INTERP_WLS, "rbf": M.INTERP_RBF, "points": M.INTERP_RBF_POINTS}[c["interp"]]
        return {"K": K, "s": c["s"], "bb_mode": M.BB_SIMPLE, "interp": interp}
    bb = c.get("bb", M.BB_INTERPOLATED)
    return {"K": c.get("K", 16), "s": c.get("s", 1.0), "bb_mode": bb, "interp": M.INTERP_WLS}


_STENCILS = {}


def _stencils(c, **over):
    rule = {**_rule(c), **over}
    key = tuple(c.get(k) for k in ("kind", "nx", "ny", "n", "phi", "geo", "scale", "hybrid")) + tuple(rule.values())
    if key not in _STENCILS:
        while len(_STENCILS) >= 8:
            _STENCILS.pop(next(iter(_STENCILS)))
        _STENCILS[key] = M.build_stencils_for(_node_set(c), **rule)
    return _STENCILS[key]


def _taus(c):
    """(tau+, tau-) of a case; tau- = 0 selects BGK."""
    if c["kind"] in ("vortex", "lattice"):
        d = 40.0 * c["scale"] / c["s"] if c["kind"] == "vortex" else float(c["d"])
        return 3.0 * U0 * d / c["re"] + 0.5, 0.0
    if c.get("model") != "bgk":
        return 1.0, 0.0
    return c["tau"], 0.5 + LAMBDA / (c["tau"] - 0.5) if c["trt"] else 0.0


def _flow(w, seed, inflow=False):
    """(rho, ux, uy) of a flow in progress: a few long modes of random phase
    (over a parabolic through-flow for the vortex street), at rest on walls."""
    rng = np.random.default_rng([77, seed])
    x0, y0, x1, y1 = w.box
    X, Y = (w.xy[:, 0] - x0) / (x1 - x0), (w.xy[:, 1] - y0) / (y1 - y0)
    out = np.zeros((w.n, 3))
    for col, amp in ((0, 5e-4), (1, 5e-3), (2, 5e-3)):
        for _ in range(4):
            kx, ky = rng.integers(1, 5, 2)
            out[:, col] += amp * rng.uniform(0.3, 1.0) * np.sin(2 * np.pi * kx * X + rng.uniform(0, 6.28)) * \
                np.cos(np.pi * ky * Y + rng.uniform(0, 6.28))
    out[:, 0] += 1.0
    if inflow:
        out[:, 1] += 4.0 * U0 * Y * (1.0 - Y)
    out[w.node_class == I.WALL, 1:] = 0.0
    eq = w.node_class == I.EQ
    out[eq] = w.eq_values[eq]
    return out


def _batch_runs(c):
    return [([1.0, 0.5, 0.25][i % 3], [1e-6, 5e-6, 2e-5][(i // 3) % 3]) for i in range(c["runs"])]


def _net_params(seed, outs):
    """He-normal weights and small biases of the 16-64-64-64-outs network, packed."""
    rng = np.random.default_rng([5, seed])
    parts = []
    for a, b in ((16, 64), (64, 64), (64, 64), (64, outs)):
        parts += [rng.normal(0.0, math.sqrt(2.0 / a), a * b), rng.normal(0.0, 0.05, b)]
    return np.concatenate(parts).astype(np.float32)


def _training_set(c, seed):
    """Features (unit scale, some at their clamps) and smooth noisy targets."""
    gen = torch.Generator(device="cuda").manual_seed(1_000_003 * seed + 17)
    X = torch.randn((c["rows"], 16), generator=gen, device="cuda").clamp_(-2.0, 4.0)
    mix = torch.randn((16, c["outs"]), generator=gen, device="cuda") * 0.3
    T = torch.tanh(X @ mix) + 0.1 * torch.randn((c["rows"], c["outs"]), generator=gen, device="cuda")
    return X.contiguous(), T.contiguous()


def _field_arrays(c, seed):
    gen = torch.Generator(device="cuda").manual_seed(1_000_003 * seed + 29)
    n = c["n"]
    r = [torch.rand(n, generator=gen, device="cuda") for _ in range(4)]
    rho, ux, uy, area = 1.0 + 1e-3 * (r[0] - 0.5), 1e-2 * (r[1] - 0.3), 1e-2 * (r[2] - 0.5), 0.5 + r[3]
    mask = (torch.rand(n, generator=gen, device="cuda") < 0.97).to(torch.uint8) if c["mask"] else None
    return rho, ux, uy, area, mask


def prepare(case, seed):
    c, kind = case, case["kind"]
    tp, tm = _taus(c) if kind not in ("train", "sums", "warm") else (1.0, 0.0)
    if kind in ("channel", "porous", "steady", "vortex"):
        w = _node_set(c)
        model = M.MODEL_BGK if kind == "vortex" or c.get("model") == "bgk" else M.MODEL_TAU1
        ctx = M.init(_stencils(c), M.Params(model, tp, tm, c.get("g", 0.0), 0.0))
        M.set_fields(ctx, _flow(w, seed, inflow=kind == "vortex"))
        M.prepare_graphs(ctx)
        return {"case": c, "ctx": ctx, "length": float(w.disks[0, 2] * 2) if kind == "vortex" else 1.0}
    if kind == "batch":
        w, runs = _node_set(c), _batch_runs(c)
        ctx = M.batch_init([_stencils(c, s=s) for s, _ in runs],
                           [M.Params(M.MODEL_TAU1, 1.0, 0.0, g, 0.0) for _, g in runs])
        M.set_fields(ctx, np.concatenate([_flow(w, 1000 * seed + i) for i in range(len(runs))], 0))
        M.prepare_graphs(ctx)
        return {"case": c, "ctx": ctx}
    if kind == "part":
        w = _node_set(c)
        part = M.Partitioned(_stencils(c), M.Params(M.MODEL_TAU1, 1.0, 0.0, c["g"], 0.0), c["parts"])
        part.set_fields(_flow(w, seed))
        return {"case": c, "part": part}
    if kind == "lattice":
        cell, eqv = I.karman_lattice(c["d"], U0)
        lat = M.Lattice(cell, M.Params(M.MODEL_BGK, tp, 0.0, 0.0, 0.0), periodic=(False, False), eq_values=eqv)
        lat.set_populations(_lattice_start(c, seed))
        return {"case": c, "lattice": lat}
    if kind == "train":
        X, T = _training_set(c, seed)
        net = M.Mlp(1, c["outs"])
        net.set_params(_net_params(seed, c["outs"]))
        return {"case": c, "net": net, "X": X, "T": T}
    if kind == "warm":
        w = _node_set(c)
        net = M.Mlp(1, c["outs"])
        net.set_params(_net_params(seed, c["outs"]))
        ctx = M.init(_stencils(c), M.Params(M.MODEL_TAU1, 1.0, 0.0, c["g"], 0.0))
        return {"case": c, "w": w, "net": net, "ctx": ctx, "X": torch.empty((w.n, 16), device="cuda")}
    rho, ux, uy, area, mask = _field_arrays(c, seed)
    need = M.reduce_scratch_doubles(c["n"])
    return {"case": c, "arrays": (rho, ux, uy, area), "mask": mask,
            "scratch": torch.empty(need, dtype=torch.float64, device="cuda"), "need": need}


def _single(a):
    """The state in its own precision."""
    return torch.from_numpy(np.ascontiguousarray(a)).to(torch.float32)


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind in ("channel", "porous"):
        ctx = state["ctx"]
        M.step(ctx, c["steps"])
        if c["model"] == "bgk":
            return [_single(M.get_populations(ctx))]
        rho, u = M.macroscopics(ctx)
        return [_single(rho), _single(u)]
    if kind == "steady":
        ctx = state["ctx"]
        taken = M.run_to_steady(ctx, 1e-12, c["window"], c["steps"], raise_on_max=False, check=c["check"])
        k = M.permeability(ctx)
        rho, u = M.macroscopics(ctx)
        return [taken, k, _single(rho), _single(u)]
    if kind == "batch":
        ctx = state["ctx"]
        M.step(ctx, c["steps"])
        k = M.batch_permeability(ctx)
        ru = _single(M.get_fields(ctx))
        return [{name: _single(v) for name, v in k.items()}, ru[:, 0], ru[:, 1:]]
    if kind == "vortex":
        ctx, forces = state["ctx"], []
        for _ in range(c["records"]):
            M.step(ctx, c["every"])
            forces.append(list(M.drag_lift(ctx, state["length"], U0)))
        return [torch.tensor(forces, dtype=torch.float32), _single(M.get_populations(ctx))]
    if kind == "part":
        part = state["part"]
        part.step(c["steps"])
        ru = _single(part.get_fields())
        return [ru[:, 0], ru[:, 1:]]
    if kind == "lattice":
        lat, forces = state["lattice"], []
        for _ in range(c["records"]):
            lat.step(c["every"])
            forces.append(list(lat.force()))
        return [torch.tensor(forces, dtype=torch.float32), _single(lat.get_populations())]
    if kind == "train":
        net, X, T = state["net"], state["X"], state["T"]
        loss = net.train(X.data_ptr(), T.data_ptr(), c["rows"], c["batch"], c["steps"], c["lr"], 12345)
        return [torch.from_numpy(net.get_params()), loss]
    if kind == "warm":
        w, ctx, net, X = state["w"], state["ctx"], state["net"], state["X"]
        L = warmstart.length_scale(w)
        M.features_for(w, L, X.data_ptr())
        cold = M.warm_start(ctx, net, X.data_ptr(), warmstart.velocity_scale(c["g"], 1.0, L),
                            warmstart.density_scale(c["g"], L) if c["outs"] == 3 else None)
        rho, u = M.macroscopics(ctx)
        return [X, cold, _single(rho), _single(u)]
    rho, ux, uy, area = state["arrays"]
    out = torch.empty(6, dtype=torch.float64, device="cuda")
    M.reduce_fields_device(rho.data_ptr(), ux.data_ptr(), uy.data_ptr(), area.data_ptr(),
                           state["mask"].data_ptr() if state["mask"] is not None else None, c["n"],
                           state["scratch"].data_ptr(), state["need"], out.data_ptr(),
                           torch.cuda.current_stream().cuda_stream)
    return [out]


# ---------------------------------------------------------------- floor counts
def _net_flops(rows, outs, backward):
    macs = 16 * 64 + 64 * 64 + 64 * 64 + 64 * outs
    # forward, then the weight gradients and the input gradients of all layers but the first
    return 2.0 * rows * (macs + (2 * macs - 16 * 64 if backward else 0))


def work(case):
    c, kind = case, case["kind"]
    if kind == "sums":
        return {"bytes": c["n"] * (16 + (1 if c["mask"] else 0)) + 48, "flops": 12.0 * c["n"]}
    if kind == "train":
        rows = c["steps"] * c["batch"]
        return {"bytes": rows * 4.0 * (16 + c["outs"]) + 3 * 8 * 9602.0, "flops": _net_flops(rows, c["outs"], True)}
    if kind == "lattice":
        cells = int(round(22.0 * c["d"])) * int(round(4.1 * c["d"]))
        steps = c["every"] * c["records"]
        return {"bytes": 73.0 * cells * steps + 72.0 * cells, "flops": 120.0 * cells * steps}
    w = _node_set(c)
    if kind == "warm":
        return {"bytes": w.n * (16.0 + 64 + 64 + 4 * c["outs"] + 24), "flops": _net_flops(w.n, c["outs"], False)}
    # per step: the stored stencil (6 K matrix entries or 8 weight rows, K indices, a kind byte), the state
    # read once and written once; equilibrium nodes write their values, lattice nodes read 9 indices
    K, tau1 = _rule(c)["K"], kind in ("steady", "batch", "part") or c.get("model") == "tau1"
    state = 4 * 3 if tau1 else 4 * 9
    rows = 6 if _rule(c)["interp"] == M.INTERP_WLS else 8
    info = M.stencils_info(_stencils(c))
    steps = c["steps"] if "steps" in c else c["every"] * c["records"]
    runs = c.get("runs", 1)
    if _rule(c)["interp"] == M.INTERP_RBF_POINTS:
        wls = 2 * state + 8 * 25 * 4 + 40 * 4 + 1  # eight stencils of 25 weights over ~40 distinct nodes
    else:
        wls = 2 * state + 4 * rows * K + 4 * K + 1
    step = info["n_wls"] * wls + info["n_lagrange"] * (2 * state + 53) + info["n_eq"] * (12 + state + 1)
    flops = (16.0 * K + 150.0) * w.n
    return {"bytes": runs * (steps * float(step) + 2 * state * w.n), "flops": runs * steps * flops}


# ------------------------------------------------------------ 64-bit arithmetic
EX = torch.tensor([0, 1, 0, -1, 0, 1, -1, -1, 1], dtype=torch.float64)
EY = torch.tensor([0, 0, 1, 0, -1, 1, 1, -1, -1], dtype=torch.float64)
WK = torch.tensor([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, dtype=torch.float64)
OPP = [0, 3, 4, 1, 2, 7, 8, 5, 6]


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _f64(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=_dev())


def _wrap(d, length, periodic):
    if not periodic:
        return d
    d = torch.where(d >= 0.5 * length, d - length, d)
    return torch.where(d < -0.5 * length, d + length, d)


def _nearest(w, K, points=None):
    """K nearest nodes of every node (or of the given points), with offsets from the point."""
    xy = _f64(w.xy)
    q = xy if points is None else points
    lx, ly = w.box[2] - w.box[0], w.box[3] - w.box[1]
    px, py = w.sides[0] == I.PERIODIC, w.sides[2] == I.PERIODIC
    # nodes sorted by x; a chunk of points looks at the strip around it
    order = torch.argsort(xy[:, 0])
    reach = 8.0 * w.h_ref * max(1.0, math.sqrt(K / 16.0))
    ext = [order]
    exx = [xy[order, 0]]
    if px:
        ext = [order, order, order]
        exx = [xy[order, 0] - lx, xy[order, 0], xy[order, 0] + lx]
    ext, exx = torch.cat(ext), torch.cat(exx)
    qo = torch.argsort(q[:, 0])
    idx = torch.empty((len(q), K), dtype=torch.int64, device=xy.device)
    step = max(64, min(2048, int(2e8 // max(1.0, len(w.xy) ** 0.5 * 60))))
    for a in range(0, len(q), step):
        rows = qo[a:a + step]
        p = q[rows]
        lo = torch.searchsorted(exx, p[:1, 0] - reach)
        hi = torch.searchsorted(exx, p[-1:, 0] + reach)
        cand = torch.unique(ext[int(lo):int(hi)])
        dx = _wrap(xy[cand, 0][None] - p[:, 0:1], lx, px)
        dy = _wrap(xy[cand, 1][None] - p[:, 1:2], ly, py)
        d2 = dx * dx + dy * dy
        # ties go to the lower node id: take a few more, sort by distance, then id (cand is ascending)
        far = torch.topk(d2, min(K + 8, len(cand)), dim=1, largest=False).indices
        far = torch.sort(far, dim=1).values
        near = torch.sort(torch.gather(d2, 1, far), dim=1, stable=True).indices[:, :K]
        idx[rows] = cand[torch.gather(far, 1, near)]
    off = torch.stack([_wrap(xy[idx, 0] - q[:, 0:1], lx, px), _wrap(xy[idx, 1] - q[:, 1:2], ly, py)], -1)
    return idx, off


def _links(w, s):
    """(link [n][9], entry fraction q [n][9]) of the departure segments that enter a solid."""
    xy = _f64(w.xy)
    n = len(xy)
    x0, y0, x1, y1 = w.box
    px, py = w.sides[0] == I.PERIODIC, w.sides[2] == I.PERIODIC
    best = torch.full((n, 9), 2.0, dtype=torch.float64, device=xy.device)
    for k in range(1, 9):
        vx, vy = -s * float(EX[k]), -s * float(EY[k])
        for side, v, dist in ((2, -vy, xy[:, 1] - y0), (3, vy, y1 - xy[:, 1]), (0, -vx, xy[:, 0] - x0),
                              (1, vx, x1 - xy[:, 0])):
            if w.sides[side] == I.SOLID and v > 0:
                t = torch.where(dist <= 1e-9 * s, torch.zeros_like(dist), dist / v)
                best[:, k] = torch.where((t < 1.0) & (t < best[:, k]), t, best[:, k])
    for cx, cy, r in np.asarray(w.disks).reshape(-1, 3):
        for ix in ((-1, 0, 1) if px else (0,)):
            for iy in ((-1, 0, 1) if py else (0,)):
                X, Y = cx + ix * (x1 - x0), cy + iy * (y1 - y0)
                if X + r + 2 * s < x0 or X - r - 2 * s > x1:
                    continue
                near = torch.nonzero((xy[:, 0] - X).abs().maximum((xy[:, 1] - Y).abs()) < r + 2 * s)[:, 0]
                rx, ry = xy[near, 0] - X, xy[near, 1] - Y
                dist = torch.sqrt(rx * rx + ry * ry)
                on = dist <= r * (1 + 1e-9)
                for k in range(1, 9):
                    vx, vy = -s * float(EX[k]), -s * float(EY[k])
                    bb, aa = rx * vx + ry * vy, vx * vx + vy * vy
                    disc = bb * bb - aa * (rx * rx + ry * ry - r * r)
                    t = (-bb - torch.sqrt(disc.clamp(min=0))) / aa
                    hit = ~on & (disc > 0) & (t >= 0) & (t < 1)
                    b = best[near, k]
                    b = torch.where(hit & (t < b), t, b)
                    best[near, k] = torch.where(on & (bb < 0), torch.zeros_like(b), b)
    link = best < 1.0
    eq = torch.as_tensor(w.node_class == I.EQ, device=xy.device)
    link[eq] = False
    return link, torch.where(link, best, torch.zeros_like(best))


def _quadratic(x, y):
    return torch.stack([torch.ones_like(x), x, y, x * x, x * y, y * y], -1)


def _operator(w, K, s, bb, interp):
    """Node set -> {"idx" [n][J], "W" [n][8][J]: the weights of direction k's value; "src": the population it
    takes; "own": links that copy the node's own population; "link", "eq"}."""
    n = w.n
    own_k = 16 if interp == M.INTERP_RBF_POINTS else K
    idx, off = _nearest(w, own_k)
    link, q = _links(w, s)
    dev = idx.device
    eq = torch.as_tensor(w.node_class == I.EQ, device=dev)
    ex, ey = EX.to(dev)[1:], EY.to(dev)[1:]
    t = torch.where(link[:, 1:], 1 - 2 * q[:, 1:], -torch.ones((), dtype=torch.float64, device=dev))  # [n][8]
    px, py = t * ex * s, t * ey * s
    use = ~link[:, 1:] if bb == M.BB_SIMPLE else torch.ones_like(link[:, 1:])
    rk = torch.sqrt((off ** 2).sum(-1).max(1).values)
    W = torch.zeros((n, 8, own_k), dtype=torch.float64, device=dev)
    if interp == M.INTERP_WLS:
        u = off / rk[:, None, None]
        g = torch.exp(-(u ** 2).sum(-1) * 2.0)
        P = _quadratic(u[..., 0], u[..., 1])
        A = torch.einsum("nja,nj,njb->nab", P, g, P)
        for a in range(0, n, 65536):
            b = slice(a, a + 65536)
            B = torch.einsum("nja,nj->naj", P[b], g[b])
            D = _quadratic(px[b] / rk[b, None], py[b] / rk[b, None])
            W[b] = D @ torch.linalg.solve(A[b], B)
    elif interp == M.INTERP_RBF:
        for k in range(8):
            W[:, k] = _phs(off, px[:, k], py[:, k])
    # the regular blocks (biquadratic Lagrange)
    r = torch.sqrt((off ** 2).sum(-1))
    h = torch.where(r > 0, r, torch.full_like(r, 1e30)).min(1).values
    lag = torch.zeros(n, dtype=torch.bool, device=dev)
    e9 = [(int(EX[m]), int(EY[m])) for m in range(9)]
    for m in range(9):
        cx, cy = e9[m][0] * h, e9[m][1] * h
        ok = ~lag & ~eq
        inside = ((px - cx[:, None]).abs() <= h[:, None] * (1 + 1e-9)) & ((py - cy[:, None]).abs() <= h[:, None] * (1 + 1e-9))
        ok &= (inside | ~use).all(1)
        rows = torch.nonzero(ok)[:, 0]
        slots = []
        for b in (-1, 0, 1):
            for a in (-1, 0, 1):
                if not len(rows):
                    break
                dx = (off[rows, :, 0] - (cx[rows] + a * h[rows])[:, None]).abs()
                dy = (off[rows, :, 1] - (cy[rows] + b * h[rows])[:, None]).abs()
                found = (dx <= 1e-9 * h[rows, None]) & (dy <= 1e-9 * h[rows, None])
                keep = found.any(1)
                slots = [x[keep] for x in slots] + [found[keep].to(torch.int8).argmax(1)]
                rows = rows[keep]
        if not len(rows):
            continue
        lag[rows] = True
        W[rows] = 0.0
        tx = px[rows] / h[rows, None] - e9[m][0]
        ty = py[rows] / h[rows, None] - e9[m][1]
        lx = [0.5 * tx * (tx - 1), (1 - tx) * (1 + tx), 0.5 * tx * (tx + 1)]
        ly = [0.5 * ty * (ty - 1), (1 - ty) * (1 + ty), 0.5 * ty * (ty + 1)]
        for i, sl in enumerate(slots):
            W[rows[:, None], torch.arange(8, device=dev)[None], sl[:, None]] += lx[i % 3] * ly[i // 3]
    if interp == M.INTERP_RBF_POINTS:
        # one stencil of 25 nodes per direction: widen to [n][8 * 25] with the weights block by block
        keep = (lag | eq)
        xy = _f64(w.xy)
        widx = torch.zeros((n, 8, 25), dtype=torch.int64, device=dev)
        wide = torch.zeros((n, 8, 25), dtype=torch.float64, device=dev)
        widx[:, :, :16], wide[:, :, :16] = idx[:, None], W
        rows = torch.nonzero(~keep)[:, 0]
        for k in range(8):
            here = rows[use[rows, k]]
            p = xy[here] + torch.stack([px[here, k], py[here, k]], -1)
            j, o = _nearest(w, 25, p)
            widx[here, k] = j
            zero = torch.zeros(len(here), dtype=torch.float64, device=dev)
            wide[here, k] = _phs(o, zero, zero)
        idx, W = widx, wide
    src = torch.arange(1, 9, device=dev).repeat(n, 1)
    opp = torch.tensor(OPP, device=dev)
    src = torch.where(link[:, 1:], opp[src], src)
    return {"idx": idx, "W": W, "src": src, "copy": ~use, "link": link, "eq": eq,
            "eqv": _f64(w.eq_values), "area": _f64(w.area)}


def _phs(off, dx, dy):
    """Cubic polyharmonic spline weights with quadratic terms at offset (dx, dy) of every stencil."""
    n, K, _ = off.shape
    out = torch.empty((n, K), dtype=torch.float64, device=off.device)
    for a in range(0, n, 16384):
        o = off[a:a + 16384]
        rk = torch.sqrt((o ** 2).sum(-1).max(1).values)[:, None]
        u, v = o[..., 0] / rk, o[..., 1] / rk
        du, dv = dx[a:a + 16384, None] / rk, dy[a:a + 16384, None] / rk
        r = torch.sqrt((u[:, :, None] - u[:, None]) ** 2 + (v[:, :, None] - v[:, None]) ** 2)
        P = _quadratic(u, v)
        A = torch.zeros((len(o), K + 6, K + 6), dtype=torch.float64, device=off.device)
        A[:, :K, :K], A[:, :K, K:], A[:, K:, :K] = r ** 3, P, P.transpose(1, 2)
        rd = torch.sqrt((u - du) ** 2 + (v - dv) ** 2)
        rhs = torch.cat([rd ** 3, _quadratic(du[:, 0], dv[:, 0])], 1)
        out[a:a + 16384] = torch.linalg.solve(A, rhs)[:, :K]
    return out


def _interpolate(op, values):
    """values [n][C] at every direction's point -> [n][8][C]; point stencils hold an index block per direction."""
    idx, W = op["idx"], op["W"]
    if idx.dim() == 3:
        return torch.einsum("nkj,nkjc->nkc", W, values[idx])
    return W @ values[idx]


def _feq(rho, ux, uy):
    ex, ey, wk = EX.to(rho.device), EY.to(rho.device), WK.to(rho.device)
    eu = ux[:, None] * ex + uy[:, None] * ey
    return wk * rho[:, None] * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * (ux * ux + uy * uy)[:, None])


def _arriving(op, f):
    """Streamed populations [n][9]."""
    n = len(f)
    g = torch.empty_like(f)
    g[:, 0] = f[:, 0]
    idx, W, src = op["idx"], op["W"], op["src"]
    for k in range(8):
        j = idx[:, k] if idx.dim() == 3 else idx
        v = (W[:, k] * f[j, src[:, k, None]]).sum(1)
        g[:, k + 1] = torch.where(op["copy"][:, k], f[torch.arange(n, device=f.device), src[:, k]], v)
    return g


def _collide(f, tp, tm, gx):
    ex, ey, wk = EX.to(f.device), EY.to(f.device), WK.to(f.device)
    rho = f.sum(1)
    ux, uy = (f @ ex) / rho + 0.5 * gx, (f @ ey) / rho
    fe = _feq(rho, ux, uy)
    d = f - fe
    dm = d[:, OPP]
    eu = ux[:, None] * ex + uy[:, None] * ey
    sp = wk * rho[:, None] * (9 * eu * ex * gx - 3 * (ux * gx)[:, None])
    sm = wk * rho[:, None] * 3 * ex * gx
    tm = tm if tm > 0 else tp
    return f - 0.5 * (d + dm) / tp - 0.5 * (d - dm) / tm + (1 - 0.5 / tp) * sp + (1 - 0.5 / tm) * sm


def _bgk_step(op, f, tp, tm, gx):
    out = _collide(_arriving(op, f), tp, tm, gx)
    e = op["eqv"]
    return torch.where(op["eq"][:, None], _feq(e[:, 0].clamp(min=1e-300), e[:, 1], e[:, 2]), out)


def _tau1_step(op, v, gx):
    """(rho, ux, uy) of the next step of the tau = 1 model."""
    n, dev = len(v), v.device
    at = _interpolate(op, v)
    at = torch.where(op["copy"][..., None], v[:, None], at)
    ex, ey, wk = EX.to(dev), EY.to(dev), WK.to(dev)
    rho = torch.zeros(n, dtype=torch.float64, device=dev)
    jx, jy = rho.clone(), rho.clone()
    for k in range(9):
        a = v if k == 0 else at[:, k - 1]
        s = torch.zeros(n, dtype=torch.int64, device=dev) if k == 0 else op["src"][:, k - 1]
        x, y, wq = ex[s], ey[s], wk[s]
        r, u, t = a[:, 0], a[:, 1], a[:, 2]
        eu = x * u + y * t
        f = wq * r * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * (u * u + t * t))
        f = f + 0.5 * wq * r * (3 * x * gx - 3 * u * gx + 9 * eu * x * gx)
        rho, jx, jy = rho + f, jx + f * ex[k], jy + f * ey[k]
    out = torch.stack([rho, jx / rho + 0.5 * gx, jy / rho], 1)
    return torch.where(op["eq"][:, None], op["eqv"], out)


def _wall_force(op, f, s):
    """Momentum exchange over the links of the next streaming step, relative to rest."""
    g = _arriving(op, f)
    a = op["area"] / (s * s)
    F = [0.0, 0.0]
    for k in range(1, 9):
        m, kp = op["link"][:, k], OPP[k]
        v = 2 * ((g[:, k] - float(WK[k])) * a)[m].sum()
        F[0] += float(v) * float(EX[kp])
        F[1] += float(v) * float(EY[kp])
    return F


def _porous_numbers(w, v, g):
    """The observables of the porous flow from (rho, ux, uy)."""
    a = _f64(w.area) * torch.as_tensor(w.node_class != I.EQ, device=v.device)
    sx, total = float((v[:, 1] * a).sum()), float(a.sum())
    us = sx / ((w.box[2] - w.box[0]) * (w.box[3] - w.box[1]))
    return {"k": us / 6.0 / g, "u_superficial": us, "u_intrinsic": sx / total,
            "tortuosity": float((torch.hypot(v[:, 1], v[:, 2]) * a).sum()) / sx}


def _lattice_start(c, seed):
    cell, eqv = I.karman_lattice(c["d"], U0)
    ny, nx = cell.shape
    rng = np.random.default_rng([91, seed])
    Y, X = np.mgrid[0:ny, 0:nx] / max(nx, ny)
    v = 4 * U0 * (Y * max(nx, ny) / (ny - 1)) * (1 - Y * max(nx, ny) / (ny - 1))
    ux = v * (1 + 0.1 * np.sin(6.28 * rng.integers(1, 9) * X + rng.uniform(0, 6.28)))
    uy = 0.1 * v * np.sin(6.28 * rng.integers(1, 9) * X + rng.uniform(0, 6.28))
    rho = 1 + 1e-3 * np.sin(6.28 * rng.integers(1, 5) * X + rng.uniform(0, 6.28))
    rho, ux, uy = (np.where(cell == 1, z, a).ravel() for z, a in ((1.0, rho), (0.0, ux), (0.0, uy)))
    ex, ey, wk = EX.numpy(), EY.numpy(), WK.numpy()
    eu = ux[:, None] * ex + uy[:, None] * ey
    return wk * rho[:, None] * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * (ux * ux + uy * uy)[:, None])


def _exact_lattice(c, seed):
    cell, eqv = I.karman_lattice(c["d"], U0)
    ny, nx = cell.shape
    dev = _dev()
    solid = torch.as_tensor(cell == 1, device=dev)
    eq = torch.as_tensor(cell == 2, device=dev).reshape(-1)
    e = _f64(eqv).reshape(-1, 3)
    feq = _feq(e[:, 0], e[:, 1], e[:, 2])
    start = f = _f64(_lattice_start(c, seed))
    tp, tm = _taus(c)
    bounce = []
    for k in range(9):
        outside = torch.zeros((ny, nx), dtype=torch.bool, device=dev)
        x, y = int(EX[k]), int(EY[k])
        if x:
            outside[:, 0 if x > 0 else -1] = True
        if y:
            outside[0 if y > 0 else -1] = True
        bounce.append(outside | torch.roll(solid, (y, x), (0, 1)))
    fluid = ~solid & ~eq.reshape(ny, nx)
    forces = []
    for i in range(c["every"] * c["records"]):
        P = f.reshape(ny, nx, 9)
        g = torch.stack([torch.where(bounce[k], P[..., OPP[k]], torch.roll(P[..., k], (int(EY[k]), int(EX[k])), (0, 1)))
                         for k in range(9)], -1).reshape(-1, 9)
        f = torch.where(eq[:, None], feq, _collide(g, tp, tm, 0.0))
        f = torch.where(solid.reshape(-1, 1), start, f)
        if (i + 1) % c["every"] == 0:
            F = [0.0, 0.0]
            for k in range(1, 9):
                m = fluid & torch.roll(solid, (int(EY[k]), int(EX[k])), (0, 1))
                v = 2 * float((f.reshape(ny, nx, 9)[..., OPP[k]][m] - float(WK[k])).sum())
                F = [F[0] + v * float(EX[OPP[k]]), F[1] + v * float(EY[OPP[k]])]
            forces.append(F)
    return [torch.tensor(forces, dtype=torch.float64), f]


def _unpack(p, outs):
    parts, o = [], 0
    for a, b in ((16, 64), (64, 64), (64, 64), (64, outs)):
        parts += [p[o:o + a * b].reshape(a, b), p[o + a * b:o + a * b + b]]
        o += a * b + b
    return parts


def _network(p, x, outs):
    q = _unpack(p, outs)
    for i in range(3):
        x = torch.relu(x @ q[2 * i] + q[2 * i + 1])
    return x @ q[6] + q[7]


def _minibatch(n, batch, seed, step):
    """The counter-based draw of a minibatch's rows: a splitmix64 hash of (seed, step, row) modulo n."""
    u = lambda v: np.uint64(v & (2 ** 64 - 1))  # noqa: E731
    with np.errstate(over="ignore"):
        z = u(seed) ^ u(step * 0xD1B54A32D192ED03) ^ (np.arange(batch, dtype=np.uint64) * u(0x9E3779B97F4A7C15))
        z = (z ^ (z >> u(30))) * u(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> u(27))) * u(0x94D049BB133111EB)
        z = z ^ (z >> u(31))
    return (z % u(n)).astype(np.int64)


def _exact_train(c, seed):
    X, T = _training_set(c, seed)
    p = _f64(_net_params(seed, c["outs"])).requires_grad_(True)
    m, v, loss = torch.zeros_like(p), torch.zeros_like(p), None
    for t in range(c["steps"]):
        rows = torch.as_tensor(_minibatch(c["rows"], c["batch"], 12345, t), device=p.device)
        e = _network(p, X[rows].double(), c["outs"]) - T[rows].double()
        loss = (e * e).sum() / c["batch"]
        (g,) = torch.autograd.grad(loss, p)
        with torch.no_grad():
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            p -= c["lr"] * (m / (1 - 0.9 ** (t + 1))) / (torch.sqrt(v / (1 - 0.999 ** (t + 1))) + 1e-8)
    return [p.detach(), float(loss)]


def _exact_features(w, L):
    xy = _f64(w.xy)
    n, dev = len(xy), xy.device
    x0, y0, x1, y1 = w.box
    lx, ly = x1 - x0, y1 - y0
    px, py = int(w.sides[0] == I.PERIODIC), int(w.sides[2] == I.PERIODIC)
    half = 0.5 * min(lx, ly)
    ell, rho = min(8 * L, half), [min(q * L, half) for q in (1.0, 2.0, 4.0, 8.0)]
    inf = float("inf")
    d1 = torch.full((n,), inf, dtype=torch.float64, device=dev)
    d2, nx, ny = d1.clone(), torch.zeros_like(d1), torch.zeros_like(d1)
    fp = [torch.full_like(d1, ell) for _ in range(4)]
    S = [torch.zeros_like(d1) for _ in range(4)]

    def take(d, ux, uy):
        nonlocal d1, d2, nx, ny
        near = d < d1
        d2 = torch.where(near, d1, torch.minimum(d2, d))
        nx, ny = torch.where(near, ux, nx), torch.where(near, uy, ny)
        d1 = torch.where(near, d, d1)

    def entry(da, db, r, sign):
        t = -sign * da - torch.sqrt(((r - db.abs()) * (r + db.abs())).clamp(min=0))
        return torch.where((db.abs() <= r) & (t >= -1e-4 * r), t.clamp(min=0), torch.full_like(t, inf))

    def lens(d, a, b):
        k = ((-d + a + b) * (d + a - b) * (d - a + b) * (d + a + b)).clamp(min=0)
        hc = torch.sqrt(k) / (2 * d)
        xa = (d * d + a * a - b * b) / (2 * d)
        xb = d - xa
        v = a * a * torch.atan2(hc, xa) - xa * hc + b * b * torch.atan2(hc, xb) - xb * hc
        v = torch.where(d <= abs(a - b), torch.full_like(d, math.pi * min(a, b) ** 2), v)
        return torch.where(d >= a + b, torch.zeros_like(d), v)

    for cx, cy, r in np.asarray(w.disks).reshape(-1, 3):
        dx0, dy0 = xy[:, 0] - cx, xy[:, 1] - cy
        if px:
            dx0 = dx0 - lx * torch.round(dx0 / lx)
        if py:
            dy0 = dy0 - ly * torch.round(dy0 / ly)
        for ix in range(-px, px + 1):
            for iy in range(-py, py + 1):
                dx, dy = dx0 + ix * lx, dy0 + iy * ly
                dist = torch.hypot(dx, dy)
                safe = dist.clamp(min=1e-300)
                take(dist - r, dx / safe, dy / safe)
                for i, (a, b, sg) in enumerate(((dx, dy, 1), (dx, dy, -1), (dy, dx, 1), (dy, dx, -1))):
                    fp[i] = torch.minimum(fp[i], entry(a, b, r, sg))
                for j in range(4):
                    S[j] += lens(safe, rho[j], r)
    one, zero = torch.ones_like(d1), torch.zeros_like(d1)
    walls = ((0, xy[:, 0] - x0, one, zero, 1), (1, x1 - xy[:, 0], -one, zero, 0), (2, xy[:, 1] - y0, zero, one, 3),
             (3, y1 - xy[:, 1], zero, -one, 2))
    for side, h, ux, uy, ray in walls:
        if w.sides[side] != I.SOLID:
            continue
        take(h, ux, uy)
        fp[ray] = torch.minimum(fp[ray], h.clamp(min=0))
        for j in range(4):
            a = rho[j]
            hc = torch.sqrt(((a - h) * (a + h)).clamp(min=0))
            seg = a * a * torch.atan2(hc, h) - h * hc
            S[j] += torch.where(h >= a, zero, torch.where(h <= -a, zero + math.pi * a * a, seg))
    d1, d2 = (torch.where(torch.isfinite(d), d, 4 * L * one) for d in (d1, d2))
    phi = 1 - float(np.sum(math.pi * np.asarray(w.disks).reshape(-1, 3)[:, 2] ** 2)) / (lx * ly)
    yy = xy[:, 1] - y0
    return torch.stack([(d1 / L).clamp(0, 4), nx, ny, (d2 / L).clamp(0, 4)] + [f / L for f in fp] +
                       [(fp[2] * fp[3] / (L * L)).clamp(max=16), ((fp[2] + fp[3]) / L).clamp(max=8)] +
                       [1 - S[j] / (math.pi * rho[j] ** 2) for j in range(4)] +
                       [one * phi, 4 * yy * (ly - yy) / (ly * ly)], 1)


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "lattice":
        return _exact_lattice(c, seed)
    if kind == "train":
        return _exact_train(c, seed)
    if kind == "sums":
        rho, ux, uy, area, mask = (a.double() if a is not None else None for a in _field_arrays(c, seed))
        a = area * mask if mask is not None else area
        q = ux * ux + uy * uy
        return [torch.stack([(b * a).sum() for b in (torch.ones_like(a), rho, ux, uy, torch.sqrt(q), q)])]
    w = _node_set(c)
    if kind == "warm":
        L = warmstart.length_scale(w)
        X = _exact_features(w, L)
        Y = _network(_f64(_net_params(seed, c["outs"])), X, c["outs"])
        u = warmstart.velocity_scale(c["g"], 1.0, L) * Y[:, :2]
        rho = torch.ones(w.n, dtype=torch.float64, device=X.device)
        if c["outs"] == 3:
            d = warmstart.density_scale(c["g"], L) * Y[:, 2]
            a = _f64(w.area)
            rho = rho + d - (d * a).sum() / a.sum()
        return [X, None, rho, u]
    rule = _rule(c)
    if kind == "batch":
        runs = _batch_runs(c)
        ops = {s: _operator(w, rule["K"], s, rule["bb_mode"], rule["interp"]) for s in {s for s, _ in runs}}
        ks, vs = [], []
        for i, (s, g) in enumerate(runs):
            v = _f64(_flow(w, 1000 * seed + i))
            for _ in range(c["steps"]):
                v = _tau1_step(ops[s], v, g)
            ks.append(_porous_numbers(w, v, g))
            vs.append(v)
        v = torch.cat(vs)
        return [{name: torch.tensor([k[name] for k in ks], dtype=torch.float64) for name in ks[0]}, v[:, 0], v[:, 1:]]
    op = _operator(w, rule["K"], rule["s"], rule["bb_mode"], rule["interp"])
    v = _f64(_flow(w, seed, inflow=kind == "vortex"))
    tp, tm = _taus(c)
    g = c.get("g", 0.0)
    if kind in ("steady", "part") or c.get("model") == "tau1":
        for _ in range(c["steps"]):
            v = _tau1_step(op, v, g)
        fields = [v[:, 0], v[:, 1:]]
        return [None, _porous_numbers(w, v, g)] + fields if kind == "steady" else fields
    f = _feq(v[:, 0], v[:, 1], v[:, 2])
    if kind != "vortex":
        for _ in range(c["steps"]):
            f = _bgk_step(op, f, tp, tm, g)
        return [f]
    forces, den = [], U0 * U0 * float(w.disks[0, 2] * 2) / c["s"]
    for _ in range(c["records"]):
        for _ in range(c["every"]):
            f = _bgk_step(op, f, tp, tm, g)
        F = _wall_force(op, f, c["s"])
        forces.append(F + [2 * F[0] / den, 2 * F[1] / den])
    return [torch.tensor(forces, dtype=torch.float64), f]
