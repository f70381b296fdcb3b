"""Performance cases: the work users of this library have it do, through its public entry points.

A case is one call (or one training step) with what a program has in hand
beforehand: a plan or batch, and grids already on the GPU.  The listed cases
span the smallest calls, ordinary ones and the largest; each storage type and
engine used in earnest; forward sweeps, convergence-checked sweeps, batches,
and gradients.  `draw` gives more cases of the same ranges.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2605_07954_gb300 import Batch, Plan, StencilFn, adjoint, inputs

TAPS = {"heat5": 5, "box9": 9, "star9": 9, "box25": 25, "star13": 13, "box49": 49}
RADIUS = {"heat5": 1, "box9": 1, "star9": 2, "box25": 2, "star13": 3, "box49": 3}
TORCH_DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}

# Multiply-adds of one sweep a drawn case may ask for (the listed 8192^2 box sweep).
MAX_MACS = 8192 * 8192 * 200 * 9
MAX_POINTS = 16384 * 16384


def _sweep(name, pattern, ny, nx, T, dtype="f32", boundary="zero", compute="auto"):
    return {"name": name, "kind": "sweep", "pattern": pattern, "ny": ny, "nx": nx, "T": T, "dtype": dtype,
            "boundary": boundary, "compute": compute}


def listed():
    return [
        # A small ragged grid advanced a few steps: what launch and exchange latency cost.
        _sweep("small_star13", "star13", 130, 517, 20),
        # Heat diffusion on the standard small grid.
        _sweep("heat_512", "heat5", 512, 512, 100),
        # A long heat run on a grid too large for one cluster and too small to fill the chip.
        _sweep("heat_1024", "heat5", 1024, 1024, 1000),
        # The two large FP32 sweeps the library is benchmarked on: 9-point box and radius-3 star.
        _sweep("box9_8192", "box9", 8192, 8192, 200),
        _sweep("star13_8192", "star13", 8192, 8192, 200),
        # The dense 7x7 box on the largest grid, full FP32 precision.
        _sweep("box49_16384", "box49", 16384, 16384, 20),
        # The same with BF16 storage and the tensor-core engine.
        _sweep("box49_tc_16384", "box49", 16384, 16384, 20, dtype="bf16", compute="tc_bf16"),
        # A grid with odd sides stored in BF16 (image-like data of any width).
        _sweep("box9_odd_bf16", "box9", 4001, 5003, 64, dtype="bf16"),
        # Many independent grids of uneven size in one call.
        {"name": "batch_256", "kind": "batch", "n": 256, "lo": 64, "hi": 2048, "T": 200},
        # Gradient of a long heat run with respect to the initial state and the weights.
        {"name": "adjoint_heat_4096", "kind": "adjoint", "pattern": "heat5", "ny": 4096, "nx": 4096, "T": 128,
         "boundary": "zero"},
        # One training step of a learnable star on a ragged medium grid: forward, loss gradient, backward.
        {"name": "train_star13", "kind": "train", "pattern": "star13", "ny": 1000, "nx": 1022, "T": 32,
         "boundary": "zero"},
        # A periodic sweep with a convergence check every 20 steps.
        {"name": "residual_box9_2048", "kind": "residual", "pattern": "box9", "ny": 2048, "nx": 2048, "T": 200,
         "m": 20, "boundary": "periodic"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sides(rng, lo, hi, even):
    """Two sides spread over [lo, hi] in logarithm, at most a factor of 4 apart, often multiples of 8."""
    ny = _log_int(rng, lo, hi)
    nx = min(hi, max(lo, int(round(ny * math.exp(rng.uniform(-math.log(4), math.log(4)))))))
    if even or rng.random() < 0.5:
        ny, nx = max(8, ny // 8 * 8), max(8, nx // 8 * 8)
    return ny, nx


def _steps(rng, points, macs, lo, hi, cap):
    """Steps spread over [lo, hi] in logarithm, no more than the work cap allows."""
    return max(1, min(_log_int(rng, lo, hi), int(cap // (points * macs))))


def draw(rng: random.Random):
    kind = rng.choices(["sweep", "tc", "batch", "adjoint", "train", "residual"], [10, 2, 1, 2, 2, 2])[0]
    boundary = rng.choices(["zero", "periodic"], [3, 1])[0]
    if kind == "sweep":
        pattern = rng.choice(["heat5", "box9", "star9", "box25", "star13", "box49"])
        ny, nx = _sides(rng, 96, 16384, False)
        return {"kind": "sweep", "pattern": pattern, "ny": ny, "nx": nx,
                "T": _steps(rng, ny * nx, TAPS[pattern], 16, 1000, MAX_MACS),
                "dtype": rng.choices(["f32", "bf16", "f16"], [4, 2, 1])[0], "boundary": boundary, "compute": "auto"}
    if kind == "tc":
        dtype = rng.choice(["bf16", "f32"])
        ny, nx = _sides(rng, 1024, 16384, True)
        return {"kind": "sweep", "pattern": "box49", "ny": ny, "nx": nx,
                "T": _steps(rng, ny * nx, 49, 8, 200, MAX_MACS), "dtype": dtype, "boundary": "zero",
                "compute": "tc_bf16" if dtype == "bf16" else "tc_tf32"}
    if kind == "batch":
        return {"kind": "batch", "n": 2 * _log_int(rng, 8, 128), "lo": 64, "hi": _log_int(rng, 256, 2048),
                "T": _log_int(rng, 20, 200)}
    if kind == "adjoint":
        pattern = rng.choice(["heat5", "box9", "star13"])
        ny, nx = _sides(rng, 256, 4096, False)
        return {"kind": "adjoint", "pattern": pattern, "ny": ny, "nx": nx, "T": _log_int(rng, 16, 128),
                "boundary": boundary}
    if kind == "train":
        pattern = rng.choice(["heat5", "box9", "star13", "box49"])
        ny, nx = _sides(rng, 128, 2048, False)
        return {"kind": "train", "pattern": pattern, "ny": ny, "nx": nx, "T": _log_int(rng, 8, 64),
                "boundary": boundary}
    pattern = rng.choice(["heat5", "box9", "star13"])
    ny, nx = _sides(rng, 256, 8192, False)
    m = _log_int(rng, 5, 50)
    return {"kind": "residual", "pattern": pattern, "ny": ny, "nx": nx, "m": m,
            "T": max(m, _steps(rng, ny * nx, TAPS[pattern], 50, 400, MAX_MACS)), "boundary": boundary}


# ---- inputs ------------------------------------------------------------------------

def _weights(pattern, seed):
    if pattern == "heat5":
        return inputs.heat_weights(0.2)
    return inputs.random_weights("star" if pattern.startswith("star") else "box", RADIUS[pattern], seed=seed)


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _field(ny, nx, seed, stream=0, dtype=torch.float32):
    """A uniform [0, 1) field, as the diffusion workloads use."""
    g = torch.Generator(device=_device())
    g.manual_seed(seed * 100003 + stream)
    return torch.rand((ny, nx), generator=g, device=_device(), dtype=torch.float32).to(dtype)


def _batch_spec(case, seed):
    """(side, weights) of every grid: sides spread log-uniformly, half 5-point stars and half 9-point boxes."""
    sides, kinds = inputs.batch_spec(case["n"], case["lo"], case["hi"], seed=0)
    return [(int(s), inputs.random_weights("box" if k == "box9" else "star", 1, seed=seed, stream=1000 + g))
            for g, (s, k) in enumerate(zip(sides, kinds))]


def _arena(spec):
    """Offsets of the grids' outputs in one buffer (each on a 256-byte boundary), and its size."""
    offsets, total = [], 0
    for side, _ in spec:
        offsets.append(total)
        total += (side * side + 63) // 64 * 64
    return offsets, total


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        spec = _batch_spec(case, seed)
        offsets, total = _arena(spec)
        # every grid's output is a piece of one buffer, as a program with many grids allocates them
        out = torch.zeros(total, dtype=torch.float32, device=_device())
        grids = [{"x": _field(side, side, seed, 10 + g), "out": out[o:o + side * side].view(side, side),
                  "weights": w, "T": case["T"]} for g, ((side, w), o) in enumerate(zip(spec, offsets))]
        return {"case": case, "grids": grids, "out": out, "batch": Batch(grids)}
    ny, nx = case["ny"], case["nx"]
    w = _weights(case["pattern"], seed)
    x = _field(ny, nx, seed, 0, TORCH_DTYPE[case.get("dtype", "f32")])
    state = {"case": case, "x": x}
    if kind == "train":
        state["x"] = x.requires_grad_(True)
        state["w"] = torch.from_numpy(w).to(x.device).requires_grad_(True)
        state["target"] = _field(ny, nx, seed, 1)
        return state
    state["plan"] = Plan(ny, nx, w, dtype=case.get("dtype", "f32"), boundary=case["boundary"],
                         compute=case.get("compute", "auto"))
    if kind == "adjoint":
        state["grad"] = _field(ny, nx, seed, 1) - 0.5
    else:
        state["out"] = torch.empty_like(x)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "sweep":
        return state["plan"].run(state["x"], case["T"], out=state["out"])
    if kind == "residual":
        return state["plan"].run_residual(state["x"], case["T"], case["m"], out=state["out"])
    if kind == "batch":
        state["batch"].run()
        return state["out"]
    if kind == "adjoint":
        return adjoint(state["plan"], state["x"], state["grad"], case["T"])
    # train: u_T, the gradient of 0.5 ||u_T - target||^2, back to the initial state and the weights
    y = StencilFn.apply(state["x"], state["w"], case["T"], case["boundary"])
    gx, gw = torch.autograd.grad(y, (state["x"], state["w"]), y.detach() - state["target"])
    return y.detach(), gx, gw


# ---- what a pass cannot do without -----------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind == "batch":
        spec = _batch_spec(case, 0)
        points = sum(s * s for s, _ in spec)
        macs = sum(s * s * int(np.count_nonzero(w)) for s, w in spec)
        return {"bytes": 8 * points, "flops": 2 * macs * case["T"]}
    points = case["ny"] * case["nx"]
    taps = TAPS[case["pattern"]]
    elem = 4 if case.get("dtype", "f32") == "f32" else 2
    if kind in ("sweep", "residual"):
        checks = case["T"] // case["m"] if kind == "residual" else 0
        return {"bytes": 2 * elem * points + 8 * checks, "flops": 2 * taps * points * case["T"] + 3 * points * checks}
    # gradients: the states forward, the adjoint recursion, and the gradient of every weight of the square
    side = (2 * RADIUS[case["pattern"]] + 1) ** 2
    grids = 3 if kind == "adjoint" else 4
    return {"bytes": 4 * grids * points, "flops": 2 * (2 * taps + side) * points * case["T"]}


# ---- exact values (64 bits, plain torch) -----------------------------------------------

def _pad64(u, r, periodic):
    """The grid extended by r rows and columns on each side: wrapped, or zeros."""
    ny, nx = u.shape
    if periodic:
        iy = torch.arange(-r, ny + r, device=u.device) % ny
        ix = torch.arange(-r, nx + r, device=u.device) % nx
        return u[iy][:, ix]
    p = torch.zeros((ny + 2 * r, nx + 2 * r), dtype=torch.float64, device=u.device)
    p[r:r + ny, r:r + nx] = u
    return p


def _step64(u, w, periodic):
    r, (ny, nx) = w.shape[0] // 2, u.shape
    p = _pad64(u, r, periodic)
    acc = torch.zeros_like(u)
    for a in range(2 * r + 1):
        for b in range(2 * r + 1):
            if w[a, b] != 0.0:
                acc.add_(p[a:a + ny, b:b + nx], alpha=float(w[a, b]))
    return acc


def _adjoint64(states, w, lam, periodic):
    """(dL/du_0, dL/dW) from the states u_0 .. u_{T-1} and dL/du_T."""
    r, (ny, nx) = w.shape[0] // 2, lam.shape
    d = 2 * r + 1
    gw = torch.zeros((d, d), dtype=torch.float64, device=lam.device)
    flipped = np.ascontiguousarray(w[::-1, ::-1])
    for u in reversed(states):
        p = _pad64(u, r, periodic)
        for a in range(d):
            for b in range(d):
                gw[a, b] += (lam * p[a:a + ny, b:b + nx]).sum()
        lam = _step64(lam, flipped, periodic)
    return lam, gw


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        spec = _batch_spec(case, seed)
        offsets, total = _arena(spec)
        out = torch.zeros(total, dtype=torch.float64, device=_device())
        for g, ((side, w), o) in enumerate(zip(spec, offsets)):
            u, w = _field(side, side, seed, 10 + g).double(), w.astype(np.float64)
            for _ in range(case["T"]):
                u = _step64(u, w, False)
            out[o:o + side * side] = u.reshape(-1)
        return out
    ny, nx, T = case["ny"], case["nx"], case["T"]
    periodic = case["boundary"] == "periodic"
    w = _weights(case["pattern"], seed).astype(np.float64)
    u = _field(ny, nx, seed, 0, TORCH_DTYPE[case.get("dtype", "f32")]).double()
    if kind == "sweep":
        for _ in range(T):
            u = _step64(u, w, periodic)
        return u
    if kind == "residual":
        res = []
        for t in range(1, T + 1):
            v = _step64(u, w, periodic)
            if t % case["m"] == 0:
                res.append(torch.linalg.vector_norm(v - u))
            u = v
        return u, torch.stack(res)
    states = []
    for _ in range(T):
        states.append(u)
        u = _step64(u, w, periodic)
    if kind == "adjoint":
        return _adjoint64(states, w, (_field(ny, nx, seed, 1) - 0.5).double(), periodic)
    gx, gw = _adjoint64(states, w, u - _field(ny, nx, seed, 1).double(), periodic)
    return u, gx, gw
