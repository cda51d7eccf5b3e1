"""The calls a user of the library makes, as cases that can be timed and checked.

A case is one pass of the work a program does with a plan it keeps: a whole
simulation from a given initial pressure (set the fields, derive the
half-step velocity, step, have p and the velocities), a batch of uneven
simulations, a run with reflection coefficients, or one call of the learned
operator.  Sizes are those of the repository's own workloads and tests, and
generic ones around them (lengths with and without small prime factors, mixed
walls, ragged batches).

Kinds:
  run      Solver.run on one grid, 1-D to 3-D (form "fft" or "split-bf16")
  order2   Solver.run2, the second-order pressure-only form
  batch    Batch.run over independent 2-D members of uneven sizes
  reflect  ReflectionRun: the 4^d wall combinations and their weighted sum
  predict  SpectralOperator.predict
  train    one training step: loss, gradients, Adam
"""
import math

import numpy as np
import torch

from paper_2005_00322_gb300 import Solver
from paper_2005_00322_gb300.batch import Batch, ReflectionRun
from paper_2005_00322_gb300.sno import SpectralOperator

C0, RHO0, DX = 1500.0, 1000.0, 1.0e-4
LEARNED_CELLS, LEARNED_WALLS = (128, 128), (("N", "N"), ("D", "D"))
CHANNELS, MODES, LAYERS = 32, 16, 4


def listed():
    return [
        # the smallest runs: one line, every pass a launch with almost no work
        {"name": "line256", "kind": "run", "form": "fft", "cells": "256", "walls": "DD", "blobs": 1, "sigma": 4.0,
         "cfl": 0.2, "steps": 512},
        # the 2-D benchmark grid: its state stays in the L2 cache, passes are short
        {"name": "plane512", "kind": "run", "form": "fft", "cells": "512x512", "walls": "DD,NN", "blobs": 4,
         "sigma": 3.0, "cfl": 0.3, "steps": 128},
        # a 2-D grid that was not chosen as a power of two, with mixed walls
        {"name": "plane375", "kind": "run", "form": "fft", "cells": "375x300", "walls": "ND,DN", "blobs": 3,
         "sigma": 3.0, "cfl": 0.3, "steps": 64},
        # independent uneven 2-D runs (most lengths have a large prime factor), advanced together
        {"name": "batch20", "kind": "batch", "members": 20, "lo": 64, "hi": 1024, "layout": 7, "steps": 32},
        # 3-D runs on the benchmark grids: the state no longer fits the L2 cache
        {"name": "cube256", "kind": "run", "form": "fft", "cells": "256x256x256", "walls": "DD,NN,DD", "blobs": 1,
         "sigma": 3.0, "cfl": 0.3, "steps": 32},
        {"name": "cube384", "kind": "run", "form": "fft", "cells": "384x384x384", "walls": "DD,NN,DD", "blobs": 4,
         "sigma": 3.0, "cfl": 0.3, "steps": 32},
        # the same grid with every derivative as a split-precision tensor-core product
        {"name": "cube384_split", "kind": "run", "form": "split-bf16", "cells": "384x384x384", "walls": "DD,NN,DD",
         "blobs": 4, "sigma": 3.0, "cfl": 0.3, "steps": 32},
        # a 3-D grid of ordinary even lengths, mixed walls
        {"name": "cube200", "kind": "run", "form": "fft", "cells": "200x180x150", "walls": "ND,NN,DD", "blobs": 2,
         "sigma": 3.0, "cfl": 0.3, "steps": 32},
        # the pressure-only form, a 3-D box with three different lengths
        {"name": "box_order2", "kind": "order2", "cells": "256x192x128", "walls": "NN,DN,DD", "blobs": 2,
         "sigma": 3.0, "cfl": 0.3, "steps": 32},
        # walls with a reflection coefficient: 64 combinations of a 3-D grid, combined
        {"name": "reflect128", "kind": "reflect", "cells": "128x128x128", "refl": 0.4, "sigma": 3.0, "cfl": 0.3,
         "steps": 32},
        # the learned operator: a batch of predictions, and a training step
        {"name": "predict256", "kind": "predict", "batch": 256},
        {"name": "train32", "kind": "train", "batch": 32},
    ]


_SMOOTH = (64, 80, 96, 100, 108, 120, 125, 128, 144, 150, 160, 180, 192, 200, 216, 240, 243, 250, 256, 270, 288, 300,
           320, 324, 360, 375, 384, 400, 405, 432, 450, 480, 486, 500, 512, 540, 576, 600, 625, 640, 648, 675, 720,
           729, 750, 768, 800, 810, 864, 900, 960, 972, 1000, 1024)


def _length(rng, lo, hi):
    """A line length in [lo, hi]: mostly one a user would round to, else any."""
    if rng.random() < 0.6:
        ok = [n for n in _SMOOTH if lo <= n <= hi]
        if ok:
            return rng.choice(ok)
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _walls(rng, plain=False):
    u = rng.random()
    if not plain and u < 0.06:
        return "PP"
    if not plain and u < 0.12:
        return rng.choice("ND") + rng.choice("nd")     # right wall at mid-cell
    return rng.choice("ND") + rng.choice("ND")


def draw(rng):
    kind = rng.choice(["line", "plane", "plane", "cube", "cube", "order2", "batch", "reflect", "predict", "train",
                       "split"])
    if kind == "line":
        return {"kind": "run", "form": "fft", "cells": str(_length(rng, 24, 2000)), "walls": _walls(rng), "blobs": 1,
                "sigma": round(rng.uniform(2.0, 2.9), 2), "cfl": 0.2, "steps": rng.randint(200, 600)}
    if kind == "plane":
        n = [_length(rng, 64, 1024) for _ in range(2)]
        return {"kind": "run", "form": "fft", "cells": "x".join(map(str, n)),
                "walls": ",".join(_walls(rng) for _ in n), "blobs": rng.randint(1, 4),
                "sigma": round(rng.uniform(2.0, 4.0), 2), "cfl": 0.3, "steps": rng.randint(48, 128)}
    if kind == "cube" or kind == "order2":
        n = [_length(rng, 40, 256) for _ in range(3)]
        c = {"kind": "run", "form": "fft"} if kind == "cube" else {"kind": "order2"}
        c.update({"cells": "x".join(map(str, n)), "walls": ",".join(_walls(rng) for _ in n),
                  "blobs": rng.randint(1, 3), "sigma": round(rng.uniform(2.0, 4.0), 2), "cfl": 0.3,
                  "steps": rng.randint(16, 40)})
        return c
    if kind == "batch":
        return {"kind": "batch", "members": rng.randint(2, 20), "lo": 64, "hi": rng.choice([256, 512, 1024]),
                "layout": rng.randint(10, 10000), "steps": rng.randint(32, 64)}
    if kind == "reflect":
        n = [_length(rng, 40, 128) for _ in range(rng.choice([2, 3]))]
        return {"kind": "reflect", "cells": "x".join(map(str, n)), "refl": round(rng.uniform(-0.5, 0.9), 3),
                "sigma": 3.0, "cfl": 0.3, "steps": rng.randint(32, 48)}
    if kind == "split":
        n = [_length(rng, 64, 256) for _ in range(3)]
        return {"kind": "run", "form": "split-bf16", "cells": "x".join(map(str, n)),
                "walls": ",".join(_walls(rng, plain=True) for _ in n), "blobs": 2,
                "sigma": round(rng.uniform(2.0, 4.0), 2), "cfl": 0.3, "steps": rng.randint(16, 32)}
    if kind == "predict":
        return {"kind": "predict", "batch": int(round(math.exp(rng.uniform(0.0, math.log(256)))))}
    return {"kind": "train", "batch": int(round(math.exp(rng.uniform(math.log(4), math.log(32)))))}


# ---- shared helpers ----------------------------------------------------------------------------------
def _cells(case):
    return tuple(int(n) for n in case["cells"].split("x"))


def _bcs(text):
    name = {"N": "N", "D": "D", "P": "P", "n": "Nm", "d": "Dm"}
    return tuple((name[w[0]], name[w[1]]) for w in text.split(","))


def _nodes(n, bc):
    """(first, last) stored pressure node of an axis."""
    if bc[0] == "P":
        return 0, n - 1
    return (1 if bc[0] == "D" else 0), (n if bc[1] == "N" else n - 1)


def _blobs(rng, cells, count, sigma):
    """Centres at least 4 sigma from the walls where the box allows it; amplitudes in [0.5, 1]."""
    out = []
    for _ in range(count):
        centre = [rng.uniform(min(4 * sigma, 0.45 * n), n - min(4 * sigma, 0.45 * n)) for n in cells]
        out.append((centre, rng.uniform(0.5, 1.0)))
    return out


def _pressure(blobs, sigma, cells, bcs):
    """Sum of Gaussian blobs on the stored nodes (FP64 on the GPU)."""
    total = 0
    for centre, amp in blobs:
        t = torch.tensor(amp, dtype=torch.float64, device="cuda")
        for n, bc, c in zip(cells, bcs, centre):
            lo, hi = _nodes(n, bc)
            x = torch.arange(lo, hi + 1, dtype=torch.float64, device="cuda")
            t = t[..., None] * torch.exp(-((x - c) ** 2) / (2 * sigma ** 2))
        total = total + t
    return total


def _initial(case, seed):
    cells, bcs = _cells(case), _bcs(case["walls"])
    rng = np.random.default_rng(seed)
    return _pressure(_blobs(rng, cells, case["blobs"], case["sigma"]), case["sigma"], cells, bcs).float()


def _members(case):
    """Sizes and walls of a batch: they belong to the case, not to the inputs."""
    rng = np.random.default_rng(case["layout"])
    out = []
    for _ in range(case["members"]):
        cells = tuple(int(v) for v in rng.integers(case["lo"], case["hi"] + 1, 2))
        out.append((cells, tuple(("ND"[int(rng.integers(2))], "ND"[int(rng.integers(2))]) for _ in range(2))))
    return out


def _member_pressures(case, seed):
    rng = np.random.default_rng(seed)
    return [_pressure(_blobs(rng, cells, 4, 3.0), 3.0, cells, bcs).float() for cells, bcs in _members(case)]


def _reflect_pressure(case, seed):
    cells = _cells(case)
    rng = np.random.default_rng(seed)
    return _pressure(_blobs(rng, cells, 1, case["sigma"]), case["sigma"], cells, (("N", "N"),) * len(cells)).float()


def _learned_inputs(batch, seed):
    """Initial pressures as the operator is trained on: 1 to 6 blobs of width 2 to 8 cells, amplitudes in [-1, 1]."""
    rng = np.random.default_rng(seed)
    x = torch.arange(0, 129, dtype=torch.float64, device="cuda")
    y = torch.arange(1, 128, dtype=torch.float64, device="cuda")
    count = torch.tensor(rng.integers(1, 7, batch), device="cuda")
    sig, cx, cy = (torch.tensor(v, device="cuda") for v in (rng.uniform(2, 8, (batch, 6)), rng.random((batch, 6)),
                                                            rng.random((batch, 6))))
    amp = torch.tensor(rng.uniform(-1, 1, (batch, 6)), device="cuda")
    amp = amp * (torch.arange(6, device="cuda")[None] < count[:, None])
    cx, cy = 4 * sig + cx * (128 - 8 * sig), 4 * sig + cy * (128 - 8 * sig)
    gx = torch.exp(-((x - cx[..., None]) ** 2) / (2 * sig[..., None] ** 2)) * amp[..., None]
    gy = torch.exp(-((y - cy[..., None]) ** 2) / (2 * sig[..., None] ** 2))
    return torch.einsum("bix,biy->bxy", gx, gy).float().contiguous()


def _learned_weights(seed):
    """Weights of a network as it stands during training (random, scaled by fan-in)."""
    rng = np.random.default_rng(seed + 1)
    c, k = CHANNELS, MODES
    w = {"w_lift": 0.5 * rng.standard_normal(c), "b_lift": 0.05 * rng.standard_normal(c),
         "w_proj": rng.standard_normal(c) / math.sqrt(c), "b_proj": 0.01 * rng.standard_normal(1)}
    for l in range(LAYERS):
        w[f"R{l}"] = rng.standard_normal((k, k, c, c)) / c
        w[f"W{l}"] = rng.standard_normal((c, c)) / math.sqrt(c)
        w[f"b{l}"] = 0.05 * rng.standard_normal(c)
    return {n: v.astype(np.float32) for n, v in w.items()}


# ---- what a program has in hand, and one pass --------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("run", "order2"):
        p0 = _initial(case, seed)
        s = Solver(_cells(case), DX, _bcs(case["walls"]), c0=C0, rho0=RHO0, cfl=case["cfl"],
                   form=case.get("form", "fft"))
        p = torch.empty_like(p0)
        if kind == "order2":
            return {"kind": kind, "solver": s, "p0": p0, "p": p, "prev": torch.empty_like(p0),
                    "steps": case["steps"]}
        us = [torch.empty(sh, device="cuda") for sh in s.shapes[1:]]
        return {"kind": kind, "solver": s, "p0": p0, "p": p, "us": us, "steps": case["steps"]}
    if kind == "batch":
        b = Batch([dict(ncells=n, dx=DX, bc=bc, cfl=0.3, c0=C0, rho0=RHO0) for n, bc in _members(case)])
        return {"kind": kind, "batch": b, "p0": _member_pressures(case, seed), "fields": b.zeros(),
                "steps": case["steps"]}
    if kind == "reflect":
        cells = _cells(case)
        r = ReflectionRun(cells, DX, [(case["refl"], case["refl"])] * len(cells), c0=C0, rho0=RHO0, cfl=case["cfl"])
        return {"kind": kind, "run": r, "p0": _reflect_pressure(case, seed), "steps": case["steps"]}
    net = SpectralOperator(LEARNED_CELLS, LEARNED_WALLS, channels=CHANNELS, modes=MODES, layers=LAYERS)
    net.set_params(_learned_weights(seed))
    x = _learned_inputs(case["batch"], seed)
    if kind == "predict":
        return {"kind": kind, "net": net, "p0": x}
    return {"kind": kind, "net": net, "p0": x, "target": _learned_inputs(case["batch"], seed + 500009)}


def run(state):
    kind = state["kind"]
    if kind == "run":
        s, p, us = state["solver"], state["p"], state["us"]
        p.copy_(state["p0"])
        for u in us:
            u.zero_()
        s.init_velocity(p, us)
        s.run(p, us, state["steps"])
        return [p] + us
    if kind == "order2":
        s, p, prev = state["solver"], state["p"], state["prev"]
        p.copy_(state["p0"])
        s.init_prev(p, prev)
        s.run2(p, prev, state["steps"])
        return [p, prev]
    if kind == "batch":
        b, fields = state["batch"], state["fields"]
        for (p, us), p0 in zip(fields, state["p0"]):
            p.copy_(p0)
            for u in us:
                u.zero_()
        b.init_velocity(fields)
        b.run(fields, state["steps"])
        return [[p] + us for p, us in fields]
    if kind == "reflect":
        r = state["run"]
        r.set_initial_pressure(state["p0"])
        r.run(state["steps"])
        return r.pressure()
    net = state["net"]
    if kind == "predict":
        return net.predict(state["p0"])
    loss, _ = net.loss_and_grads(state["p0"], state["target"])
    net.adam(lr=1e-3)
    return {"loss": loss, "grads": net.gflat, "weights": net.flat}


# ---- the same results in 64 bits ---------------------------------------------------------------------
def _axis_modes(n, bc):
    """Wavenumbers and sampled modes of one walled axis: p on its nodes and dp/dx on the half-nodes, u on the
    half-nodes and du/dx on the nodes (cos where a field is symmetric about the left wall, else sin)."""
    l, r = bc[0], bc[1][0]
    mid = len(bc[1]) == 2
    length = (n - 0.5 if mid else n) * DX
    lo, hi = _nodes(n, bc)
    x = np.arange(lo, hi + 1) * DX
    m = n - 1 if bc[1] == "Nm" else n
    h = (np.arange(m) + 0.5) * DX
    if l == r:
        b0 = 0 if l == "N" else 1
        kp = np.pi / length * (b0 + np.arange(len(x)))
        ku = np.pi / length * ((1 - b0) + np.arange(m))
    else:
        kp = np.pi / length * (0.5 + np.arange(len(x)))
        ku = np.pi / length * (0.5 + np.arange(m))
    if l == "N":
        return (np.cos(np.outer(x, kp)), -kp * np.sin(np.outer(h, kp)), np.sin(np.outer(h, ku)),
                ku * np.cos(np.outer(x, ku)))
    return (np.sin(np.outer(x, kp)), kp * np.cos(np.outer(h, kp)), np.cos(np.outer(h, ku)),
            -ku * np.sin(np.outer(x, ku)))


def _axis_operators(n, bc):
    """(dp/dx: nodes -> half-nodes, du/dx: half-nodes -> nodes) as FP64 matrices on the GPU."""
    if bc[0] == "P":
        k = 2 * np.pi * np.fft.fftfreq(n, DX)
        f = np.fft.fft(np.eye(n), axis=0)
        dp = np.fft.ifft((1j * k * np.exp(0.5j * k * DX))[:, None] * f, axis=0).real
        du = np.fft.ifft((1j * k * np.exp(-0.5j * k * DX))[:, None] * f, axis=0).real
    else:
        p, dph, u, dun = _axis_modes(n, bc)
        dp = np.linalg.solve(p.T, dph.T).T
        du = np.linalg.solve(u.T, dun.T).T
    return torch.tensor(dp, device="cuda"), torch.tensor(du, device="cuda")


def _along(op, x, axis):
    return torch.tensordot(op, x, dims=([1], [axis])).movedim(0, axis)


def _leapfrog(cells, bcs, cfl, p0, steps):
    dt = cfl * DX / C0
    ops = [_axis_operators(n, bc) for n, bc in zip(cells, bcs)]
    p = p0.double()
    us = [dt / (2 * RHO0) * _along(dp, p, a) for a, (dp, _) in enumerate(ops)]
    for _ in range(steps):
        new = p.clone()
        for a, (dp, du) in enumerate(ops):
            us[a] = us[a] - dt / RHO0 * _along(dp, p, a)
            new -= dt * RHO0 * C0 ** 2 * _along(du, us[a], a)
        p = new
    return [p] + us


def _order2(case, p0):
    cells, bcs, dt = _cells(case), _bcs(case["walls"]), case["cfl"] * DX / C0
    ops = [(du @ dp) * (C0 * dt) ** 2 for dp, du in (_axis_operators(n, bc) for n, bc in zip(cells, bcs))]
    lap = lambda f: sum(_along(op, f, a) for a, op in enumerate(ops))  # noqa: E731
    p = p0.double()
    prev = p + 0.5 * lap(p)
    for _ in range(case["steps"]):
        p, prev = 2 * p - prev + lap(p), p
    return [p, prev]


def _reflect(case, p_full):
    """Every wall combination by its modes, p^n = p^0 cos(n theta), weighted and summed on the full lattice."""
    cells, dt, n = _cells(case), case["cfl"] * DX / C0, case["steps"]
    r = case["refl"]
    # per axis and wall pair: weight of the run with image signs (left, right), from the four basic runs
    weight = {"NN": (1 + r) ** 2 / 4, "ND": (1 + r) * (1 - r) / 4, "DN": (1 - r) * (1 + r) / 4,
              "DD": (1 - r) ** 2 / 4}
    basis = []
    for cellsn in cells:
        per = {}
        for w in weight:
            phi = _axis_modes(cellsn, (w[0], w[1]))[0]
            cnt = phi.shape[1]
            off = {"NN": 0.0, "DD": 1.0, "ND": 0.5, "DN": 0.5}[w]
            k = np.pi / (cellsn * DX) * (off + np.arange(cnt))
            inv = np.linalg.inv(phi)
            per[w] = tuple(torch.tensor(v, device="cuda") for v in (phi, inv, k))
        basis.append(per)
    out = torch.zeros([c + 1 for c in cells], dtype=torch.float64, device="cuda")
    combos = [()]
    for _ in cells:
        combos = [c + (w,) for c in combos for w in weight]
    for combo in combos:
        sl = tuple(slice(_nodes(c, (w[0], w[1]))[0], _nodes(c, (w[0], w[1]))[1] + 1) for c, w in zip(cells, combo))
        f = p_full.double()[sl]
        k2 = 0
        for a, w in enumerate(combo):
            f = _along(basis[a][w][1], f, a)
            shape = [1] * len(cells)
            shape[a] = -1
            k2 = k2 + (basis[a][w][2] ** 2).reshape(shape)
        f = f * torch.cos(2 * n * torch.asin(C0 * dt * torch.sqrt(k2) / 2))
        for a, w in enumerate(combo):
            f = _along(basis[a][w][0], f, a)
        out[sl] += math.prod(weight[w] for w in combo) * f
    return out


def _learned_basis():
    """First modes of the unnormalised cosine (type I, 129 points) and sine (type I, 127 points) transforms, forward
    and inverse."""
    n, k = 128, MODES
    j = np.arange(n + 1)
    c = 2 * np.cos(np.pi * np.outer(np.arange(k), j) / n)
    tx, ix = c.copy(), c.T / (2 * n)
    tx[:, [0, n]] /= 2
    ix[:, 0] /= 2
    s = 2 * np.sin(np.pi * np.outer(np.arange(k) + 1, np.arange(1, n)) / n)
    return [torch.tensor(v, device="cuda") for v in (tx, ix, s, s.T / (2 * n))]


def _network(w, x):
    tx, ix, ty, iy = _learned_basis()
    v = w["w_lift"][None, :, None, None] * x[:, None] + w["b_lift"][None, :, None, None]
    for l in range(LAYERS):
        spec = torch.einsum("kx,bcxy,qy->bckq", tx, v, ty)
        spec = torch.einsum("kqdc,bckq->bdkq", w[f"R{l}"], spec)
        v = (torch.einsum("xk,bckq,yq->bcxy", ix, spec, iy) + torch.einsum("dc,bcxy->bdxy", w[f"W{l}"], v)
             + w[f"b{l}"][None, :, None, None])
        if l < LAYERS - 1:
            v = torch.relu(v)
    return torch.einsum("c,bcxy->bxy", w["w_proj"], v) + w["b_proj"]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("run", "order2") and math.prod(_cells(case)) * sum(_cells(case)) * case["steps"] > 2.2e12:
        return None
    if kind == "run":
        return _leapfrog(_cells(case), _bcs(case["walls"]), case["cfl"], _initial(case, seed), case["steps"])
    if kind == "order2":
        return _order2(case, _initial(case, seed))
    if kind == "batch":
        return [_leapfrog(n, bc, 0.3, p0, case["steps"])
                for (n, bc), p0 in zip(_members(case), _member_pressures(case, seed))]
    if kind == "reflect":
        return _reflect(case, _reflect_pressure(case, seed))
    w = {n: torch.tensor(v, device="cuda").double() for n, v in _learned_weights(seed).items()}
    x = _learned_inputs(case["batch"], seed).double()
    if kind == "predict":
        rms = x.square().mean(dim=(1, 2), keepdim=True).sqrt()
        return torch.cat([_network(w, (x / rms)[i:i + 64]) * rms[i:i + 64] for i in range(0, len(x), 64)])
    for v in w.values():
        v.requires_grad_()
    loss = (_network(w, x) - _learned_inputs(case["batch"], seed + 500009).double()).square().mean()
    loss.backward()
    names = ["w_lift", "b_lift", "w_proj", "b_proj"] + [f"{n}{l}" for l in range(LAYERS) for n in "RWb"]
    g = torch.cat([w[n].grad.reshape(-1) for n in names])
    flat = torch.cat([w[n].detach().reshape(-1) for n in names])
    # first Adam step: the moments' bias corrections leave g / (|g| + eps)
    return {"loss": loss.detach().reshape(1), "grads": g, "weights": flat - 1e-3 * g / (g.abs() + 1e-8)}


# ---- what a pass cannot do without -------------------------------------------------------------------
def _fft_flops(cells, transforms):
    """Real transforms of every line of every axis: 2.5 N log2 N each."""
    return sum(transforms * 2.5 * math.prod(cells) * math.log2(2 * n) for n in cells)


def work(case):
    kind = case["kind"]
    if kind in ("run", "order2"):
        cells, steps = _cells(case), case["steps"]
        points, d = math.prod(cells), len(cells)
        if kind == "order2":
            return {"bytes": 4.0 * points * (1 + 2), "flops": steps * (_fft_flops(cells, 2) + points * (d + 2))}
        if case["form"] != "fft":
            # the two derivatives of each axis as dense products, three slices of each factor (six products)
            return {"bytes": 4.0 * points * (1 + d + 1),
                    "flops": steps * sum(2 * 2.0 * n * points * 6 for n in cells)}
        # each state field read and written once a step; the state of the small grids need not leave the chip
        per = 2 * (d + 1) * 4.0 * points if 4.0 * (d + 1) * points > 126e6 else 0.0
        return {"bytes": max(4.0 * points * (d + 2), steps * per),
                "flops": steps * (_fft_flops(cells, 2) + 4 * d * points)}
    if kind == "batch":
        cells = [n for n, _ in _members(case)]
        return {"bytes": sum(4.0 * math.prod(n) * 4 for n in cells),
                "flops": case["steps"] * sum(_fft_flops(n, 2) + 8 * math.prod(n) for n in cells)}
    if kind == "reflect":
        cells = _cells(case)
        points, d, m = math.prod(cells), len(cells), 4 ** len(cells)
        per = 2 * (d + 1) * 4.0 * points * m if 4.0 * (d + 1) * points * m > 126e6 else 0.0
        return {"bytes": 4.0 * points * 2 + case["steps"] * per,
                "flops": m * case["steps"] * (_fft_flops(cells, 2) + 4 * d * points)}
    b, c, k, x, y = case["batch"], CHANNELS, MODES, 129, 127
    layer = 2.0 * b * c * (2 * x * y * k + 2 * x * k * k) + 2.0 * b * c * c * (k * k + x * y)
    weights = 4.0 * LAYERS * (k * k * c * c + c * c + c)
    if kind == "predict":
        return {"bytes": 8.0 * b * x * y + weights, "flops": LAYERS * layer}
    # the activations of every layer are kept for the backward pass (written once, read once)
    return {"bytes": 8.0 * b * x * y + 7 * weights + 8.0 * LAYERS * b * c * x * y, "flops": 3 * LAYERS * layer}
