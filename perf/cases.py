"""Performance cases: the work a user of this framework has it do, each through its public entry points.

A pass is what a driver program does between two looks at its model: step the cells' DEMs (and the coarse step) over
one or a few coarse intervals, or the truth DEM over some steps, then read the state and the moments; a call of the
closure network; a training run.  A model goes on from pass to pass, as a user's does.  The coupled method is not
stable for ever on small grids and on cells that differ much in their ice (the Lax-Friedrichs average leaves a
checkerboard undamped), so those run the cells' DEMs alone (couple = 0); the larger and more even grids run coupled.

Models in single precision hand their floes and moments over in doubles that hold FP32 results: such outputs are
returned as float32, those of an FP64 model as they come.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2303_07819_gb300 import inputs, msdem

MOMENTS = ("n", "M", "Mu", "Mv", "I", "Iw", "area", "Muu", "Mvv", "Fdx", "Fdy", "Td")
FLOES = ("x", "y", "theta", "u", "v", "omega", "r", "h")

# floes read back whole up to this many (a driver of a larger model reads the cells' moments and the coarse state at
# every output, and the floes only for a checkpoint)
WHOLE = 300_000
FLOE_STEPS = 2_000_000 * 200      # of the largest listed case


def listed():
    return [
        # the smallest call: the periodic 100 km square, 4 x 4 cells of 16 floes, one interval of 100 steps
        {"name": "cells_4x4", "kind": "cells", "scene": "square", "nx": 4, "per_cell": 16.0, "steps": 100, "couple": 0, "fp64": False},
        # the same square in FP64 (the parity precision), two intervals
        {"name": "cells_4x4_fp64", "kind": "cells", "scene": "square", "nx": 4, "per_cell": 16.0, "steps": 200, "couple": 0, "fp64": True},
        # 32 x 32 cells, Poisson(64) power-law floes: the ordinary size, two coarse intervals
        {"name": "cells_32x32", "kind": "cells", "scene": "powerlaw", "nx": 32, "per_cell": 64.0, "steps": 200, "couple": 1, "fp64": False},
        # an output period that is no multiple of the coarse interval
        {"name": "cells_27x27_ragged", "kind": "cells", "scene": "powerlaw", "nx": 27, "per_cell": 64.0, "steps": 130, "couple": 1, "fp64": False},
        # the Sec. 4.3 scenario at the paper's size: 115,200 floes, 48 x 24 cells, compressible current
        {"name": "cells_sec43", "kind": "cells", "scene": "sec43", "nx": 48, "per_cell": 100.0, "steps": 200, "couple": 1, "fp64": False},
        # the batched workload: 128 x 128 cells, about 2.0M floes, two coarse intervals
        {"name": "cells_128x128", "kind": "cells", "scene": "batched", "nx": 128, "per_cell": 96.0, "steps": 200, "couple": 1, "fp64": False},
        # an ensemble: 4 realizations of 256 x 256 cells with few floes each, about 2.0M floes, two intervals
        {"name": "ensemble_4x256x256", "kind": "cells", "scene": "ensemble", "nx": 256, "nens": 4, "per_cell": 6.0, "steps": 200, "couple": 0,
         "fp64": False},
        # a host program that holds the floes between intervals: all of them up, one interval, all of them down
        {"name": "exchange_64x64", "kind": "exchange", "scene": "batched", "nx": 64, "per_cell": 96.0, "steps": 100, "couple": 0, "fp64": False},
        # the truth DEM beside it: 65k power-law floes, and the Sec. 4.3 floes at the paper's size
        {"name": "truth_32x32", "kind": "truth", "scene": "powerlaw", "nx": 32, "per_cell": 64.0, "steps": 20, "couple": 0, "fp64": False},
        {"name": "truth_sec43", "kind": "truth", "scene": "sec43", "nx": 48, "per_cell": 100.0, "steps": 20, "couple": 0, "fp64": False},
        # the closure network on the cells of a 256 x 256 grid, and a training run on particle-path sized data
        {"name": "infer_65536", "kind": "infer", "n": 65536},
        {"name": "train_65536", "kind": "train", "n": 65536, "batch": 1024, "epochs": 4},
    ]


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def draw(rng):
    kind = rng.choice(["cells", "cells", "cells", "cells", "cells64", "truth", "truth64", "exchange", "infer", "train"])
    if kind == "infer":
        return {"kind": kind, "n": int(_log(rng, 500, 1_000_000))}
    if kind == "train":
        return {"kind": kind, "n": int(_log(rng, 2000, 130_000)), "batch": rng.choice([256, 1000, 1024, 2048, 4096, 8192]),
                "epochs": rng.randint(1, 4)}
    if kind in ("cells64", "truth64"):
        c = {"kind": kind[:-2], "scene": rng.choice(["square", "powerlaw"]), "nx": int(_log(rng, 3, 12)),
             "per_cell": _log(rng, 8, 48), "steps": rng.randint(10, 150), "couple": 0, "fp64": True}
        c["per_cell"] = min(c["per_cell"], 16.0) if c["scene"] == "square" else c["per_cell"]
        c["steps"] = min(c["steps"], 40) if kind == "truth64" else c["steps"]
        return c
    if kind == "truth":
        return {"kind": kind, "scene": "powerlaw", "nx": int(_log(rng, 4, 64)), "per_cell": _log(rng, 16, 100),
                "steps": rng.randint(1, 40), "couple": 0, "fp64": False}
    scene = rng.choice(["powerlaw", "batched", "batched", "ensemble"])
    nx = int(_log(rng, 3, 128)) if kind == "cells" else int(_log(rng, 8, 90))
    c = {"kind": kind, "scene": scene, "nx": nx, "per_cell": _log(rng, 20, 100) if scene != "ensemble" else _log(rng, 4, 16)}
    if scene == "ensemble":
        c["nens"] = rng.randint(2, 6)
    most = FLOE_STEPS / (1.35 * c["per_cell"] * nx * nx * c.get("nens", 1))
    c["steps"] = max(1, min(rng.choice([100, 200, 300, rng.randint(1, 99), rng.randint(101, 300)]), int(most)))
    c["couple"] = 1 if scene == "powerlaw" and nx >= 24 else 0
    c["fp64"] = False
    return c


# ------------------------------------------------------------------ inputs
def _physics(dt, nx, side, couple):
    return {"rho_o": 1026.0, "Cd": 5.5e-3, "rho_a": 1.3, "Ca": 1.2e-3, "wind_x": 10.0, "wind_y": 0.0, "wind_period": 0.0,
            "rho_ice": 920.0, "E": 4.0e3, "G": 5.0e3, "eta": 1.0e4 * dt, "mu": 0.3, "h_ref": 1.0, "inertia_half": 0,
            "couple": couple, "N0": 100, "n_t": 10, "uo_x": 0.0, "uo_y": 0.0, "nx": nx, "ny": nx, "Lx": nx * side, "Ly": nx * side}


def _counts(case, ncell):
    """Floes per cell: a property of the case, so that every seed fills the same layout with other floes."""
    per_cell, scene = case["per_cell"], case["scene"]
    rng = np.random.default_rng([case["nx"], int(1000 * per_cell)])
    if scene == "square":
        return np.full(ncell, int(round(per_cell)))
    if scene == "powerlaw":
        return np.maximum(rng.poisson(per_cell, ncell), 1)
    lo, hi = (1, 64) if scene == "ensemble" else (8, 1024)
    return np.clip(np.rint(per_cell * np.exp(0.69 * rng.standard_normal(ncell))), lo, hi).astype(np.int64)


def _place(gen, counts, side, r_range, flat, inside):
    """Floes of every cell without overlap, the largest first, each at the first of 32 random places that is free under
    the cell-periodic metric (inside: wholly within its cell), or shrunk into the roomiest.  Radii follow p(r) ~ r^-2
    (flat: uniform), scaled to 55 % cover where they hold more.  Returns cell, x, y, r (x, y within the cell)."""
    dev = torch.device("cuda")
    order = np.argsort(-counts, kind="stable")
    cs = counts[order]
    n_max, C = int(cs[0]), len(cs)
    u = torch.rand(C, n_max, generator=gen, device=dev)
    a, b = r_range
    R = a + u * (b - a) if flat else 1.0 / (1.0 / a - u * (1.0 / a - 1.0 / b))
    held = torch.arange(n_max, device=dev)[None, :] < torch.from_numpy(cs).to(dev)[:, None]
    R = torch.where(held, R, 0.0)
    cover = math.pi * (R * R).sum(1, keepdim=True) / side ** 2
    R = (R * torch.clamp(torch.sqrt(0.55 / cover), max=1.0)).sort(1, descending=True).values
    P = torch.zeros(C, n_max, 2, device=dev)
    live = np.searchsorted(-cs, -np.arange(1, n_max + 1), side="right")   # cells with more than k floes
    for k in range(n_max):
        m = int(live[k])
        c = torch.rand(m, 32, 2, generator=gen, device=dev)
        rk = R[:m, k]
        c = rk[:, None, None] + c * (side - 2.0 * rk[:, None, None]) if inside else c * side
        if k:
            d = c[:, :, None, 0] - P[:m, None, :k, 0]
            e = c[:, :, None, 1] - P[:m, None, :k, 1]
            d, e = d - side * torch.round(d / side), e - side * torch.round(e / side)
            room = (torch.sqrt(d * d + e * e) - R[:m, None, :k]).amin(2)
            free = room >= 1.0005 * rk[:, None]
            pick = torch.where(free.any(1), free.to(torch.int8).argmax(1), room.argmax(1))
            got = room.gather(1, pick[:, None])[:, 0]
            R[:m, k] = torch.minimum(rk, torch.clamp(0.999 * got, min=0.02 * a))
        else:
            pick = torch.zeros(m, dtype=torch.int64, device=dev)
        P[:m, k] = c[torch.arange(m, device=dev), pick]
    at = torch.nonzero(held)
    cell = torch.from_numpy(order).to(dev)[at[:, 0]]
    by = torch.argsort(cell, stable=True)
    at, cell = at[by], cell[by]
    pos, rad = P[at[:, 0], at[:, 1]].double(), R[at[:, 0], at[:, 1]].double()
    return cell, pos[:, 0], pos[:, 1], rad


def _scene(case, seed):
    """(params, floes, dt): floes as the host arrays the library takes."""
    scene, nx = case["scene"], case["nx"]
    rng = np.random.default_rng([seed, 7])
    if scene == "sec43":
        s = inputs.scenario4x(3, nfx=nx * 10, nfy=nx * 5, nx=nx, ny=nx // 2)
        f = dict(s["floes"])
        n = f["x"].shape[0]
        # no two alike: radii a little below the packing, places and thicknesses a little off the lattice
        f["r"] = f["r"] * rng.uniform(0.85, 0.97, n)
        gap = 2.0 / (nx * 5)
        f["x"] = np.mod(f["x"] + gap * rng.uniform(-0.015, 0.015, n), 4.0)
        f["y"] = np.mod(f["y"] + gap * rng.uniform(-0.015, 0.015, n), 2.0)
        f["h"] = rng.uniform(0.8, 1.2, n)
        return dict(s["params"], couple=case["couple"]), f, s["dt"]
    nens = case.get("nens", 1)
    side = 12.5e3 if scene == "powerlaw" else 25e3
    dt = 10.0 if scene == "square" else 5.0
    p = _physics(dt, nx, side, case["couple"])
    if scene == "square":
        p.update(Ca=0.0, wind_x=0.0, modes=inputs.psi_sin_sin_modes(0.1, p["Lx"]))
    else:
        p.update(modes=inputs.random_modes(rng, 8, p["Lx"], p["Ly"], 0.1), wind_period=0.0 if scene == "powerlaw" else 6 * 3600.0)
    if nens > 1:
        p["nens"] = nens
    counts = _counts(case, nens * nx * nx)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    cell, px, py, r = _place(gen, counts, side, (1000.0, 2500.0) if scene == "square" else (200.0, 3000.0),
                             scene == "square", case["kind"] == "truth")
    n = r.shape[0]
    x = (cell % nx).double() * side + px
    y = torch.div(cell, nx, rounding_mode="floor").double() * side + py
    s2 = math.log(1.0 + (0.5 / 1.5) ** 2)
    h = torch.exp(math.sqrt(s2) * torch.randn(n, generator=gen, device="cuda", dtype=torch.float64) + math.log(1.5) - 0.5 * s2)
    z = np.zeros(n)
    f = {"x": x.cpu().numpy(), "y": y.cpu().numpy(), "theta": z, "u": z, "v": z, "omega": z, "r": r.cpu().numpy(),
         "h": np.ones(n) if scene == "square" else h.cpu().numpy()}
    return p, f, dt


def _samples(n, seed):
    """Features and targets of n cells with the closure data's spreads, the network's normalisation and its weights."""
    g = torch.Generator().manual_seed(seed)
    sd = torch.tensor([150.0, 0.1, 0.1, 1e-5, 4e-3, 4e-3, 0.1, 0.1, 1e-7, 2e-6, 7.0, 7.0, 5e-6, 5e-6, 1e-10, 1e-6])
    mu = torch.tensor([750.0, 0.05, -0.02, 0.0, 5e-3, 5e-3, 0.0, 0.0, 0.0, 0.0, 3.0, 1.0, 1e-6, -1e-6, 0.0, 0.0])
    z = torch.randn(n, 16, generator=g)
    t = torch.stack([z[:, 12] + 0.3 * torch.tanh(z[:, 1] - z[:, 6]), z[:, 13] + 0.3 * torch.tanh(z[:, 2] - z[:, 7]),
                     z[:, 14] + 0.2 * torch.sin(z[:, 9]), 0.5 * z[:, 15] - 0.5 * torch.tanh(z[:, 4])], 1)
    y_sd = torch.tensor([5e-6, 5e-6, 1e-10, 1e-6])
    norm = {"mu_x": mu.numpy(), "sd_x": sd.numpy(), "mu_y": np.zeros(4, np.float32), "sd_y": y_sd.numpy()}
    return (mu + sd * z), y_sd * (t + 0.1 * torch.randn(n, 4, generator=g)), norm, inputs.mlp_init(seed)


# ------------------------------------------------------------------- a pass
def prepare(case, seed):
    if case["kind"] in ("infer", "train"):
        X, Y, norm, w = _samples(case["n"], seed)
        if case["kind"] == "infer":
            net = msdem.MLP(w, norm)
            return {"case": case, "net": net, "X": X.cuda(), "Y": torch.empty(case["n"], 4, device="cuda")}
        return {"case": case, "net": msdem.MLP(w, norm, max_batch=case["batch"]), "X": X.numpy(), "Y": Y.numpy(), "seed": seed + 1}
    p, floes, dt = _scene(case, seed)
    m = msdem.Model(p, floes, msdem.MS_FP64 if case["fp64"] else msdem.MS_FP32)
    return {"case": case, "m": m, "dt": dt, "floes": floes if case["kind"] == "exchange" else None}


def _as_held(case, a):
    return a if case["fp64"] else torch.from_numpy(a).to(torch.float32)


def _columns(case, mom):
    mom = _as_held(case, mom)
    return {k: mom[:, i] for i, k in enumerate(MOMENTS)}


def run(state):
    case = state["case"]
    if case["kind"] == "infer":
        state["net"].forward_device(state["X"].data_ptr(), case["n"], state["Y"].data_ptr())
        return state["Y"]
    if case["kind"] == "train":
        losses = state["net"].train(state["X"], state["Y"], case["epochs"], case["batch"], 2e-3, state["seed"])
        return {"loss": losses.astype(np.float32), "params": {k: v.astype(np.float32) for k, v in state["net"].params().items()}}
    m = state["m"]
    if case["kind"] == "truth":
        m.truth_step(state["dt"], case["steps"])
        return {"floes": {k: _as_held(case, v) for k, v in m.truth_floes().items()}, "moments": _columns(case, m.truth_moments())}
    if case["kind"] == "exchange":
        m.set_floes(state["floes"])
        m.step(state["dt"], case["steps"])
        state["floes"] = m.floes()
        return {"floes": {k: _as_held(case, v) for k, v in state["floes"].items()}, "moments": _columns(case, m.moments())}
    m.step(state["dt"], case["steps"])
    out = {"moments": _columns(case, m.moments())}
    if case["couple"] and case["steps"] >= 100:
        c = m.coupling()
        out["q"], out["targets"] = _as_held(case, c["q"]), _as_held(case, c["targets"])
    if m.n <= WHOLE:
        out["floes"] = {k: _as_held(case, v) for k, v in m.floes().items()}
    return out


# ---------------------------------------------------------------- its work
def _size(case):
    if case["scene"] == "sec43":
        return case["nx"] * 10 * case["nx"] * 5, case["nx"] * (case["nx"] // 2)
    nc = case["nx"] ** 2 * case.get("nens", 1)
    mean = case["per_cell"] * (math.exp(0.5 * 0.69 ** 2) if case["scene"] in ("batched", "ensemble") else 1.0)
    return int(mean * nc), nc


def work(case):
    if case["kind"] == "infer":
        return {"bytes": case["n"] * 80, "flops": case["n"] * 2 * (16 * 128 + 2 * 128 * 128 + 128 * 4)}
    if case["kind"] == "train":
        k = case["n"] * case["epochs"]
        return {"bytes": case["n"] * 80 + k * 80, "flops": k * 6 * (16 * 128 + 2 * 128 * 128 + 128 * 4)}
    n, nc = _size(case)
    word = 8 if case["fp64"] else 4
    # a floe's state in and out, once a pass, and the cells' moments; a floe-step: drag, Euler and about two contacts
    return {"bytes": n * 15 * word + nc * 12 * 8, "flops": n * case["steps"] * 200}


# ------------------------------------------------- the same in 64 bits, plain
def exact(case, seed):
    if case["kind"] == "train":
        return None       # sums of gradients in BF16 products over many updates: no one value
    if case["kind"] == "infer":
        X, _, norm, w = _samples(case["n"], seed)
        t = lambda a: torch.as_tensor(np.asarray(a, np.float32).astype(np.float64)).cuda()  # noqa: E731
        z = (X.cuda().double() - t(norm["mu_x"])) / t(norm["sd_x"])
        for i in (1, 2, 3):
            z = torch.tanh(z @ t(w["W%d" % i]).T + t(w["b%d" % i]))
        return t(norm["mu_y"]) + t(norm["sd_y"]) * (z @ t(w["W4"]).T + t(w["b4"]))
    p, floes, dt = _scene(case, seed)
    d = _Dem(p, floes, dt, case["kind"] == "truth")
    for _ in range(case["steps"]):
        d.step()
    floes = {k: v.cpu().numpy() for k, v in d.state().items()}
    mom = d.moments()
    moments = {k: mom[:, i].cpu().numpy() for i, k in enumerate(MOMENTS)}
    if case["kind"] != "cells":
        return {"floes": floes, "moments": moments}
    out = {"moments": moments}
    if case["couple"] and case["steps"] >= 100:
        out["q"], out["targets"] = d.q.cpu().numpy(), d.tgt.cpu().numpy()
    if floes["x"].shape[0] <= WHOLE:
        out["floes"] = floes
    return out


class _Dem:
    """The method in FP64 torch operations: all pairs of a cell (or of the domain) whose distance allows a contact
    within the next steps, Eq. 2.2, drag, Euler, gradual updates, the Lax-Friedrichs step."""

    EVERY = 10      # steps between two searches for pairs

    def __init__(self, p, floes, dt, truth):
        self.p, self.dt, self.truth, self.steps = p, dt, truth, 0
        self.f = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda().double().clone() for k, v in floes.items()}
        self.nx, self.ny, self.nens = p["nx"], p["ny"], p.get("nens", 1)
        self.nc = self.nx * self.ny * self.nens
        self.dX, self.dY = p["Lx"] / self.nx, p["Ly"] / self.ny
        self.Ly = p["Ly"] * self.nens
        f = self.f
        f["x"], f["y"] = torch.remainder(f["x"], p["Lx"]), torch.remainder(f["y"], self.Ly)
        self.cell = self._cells()
        if truth:
            self.px, self.py = p["Lx"], p["Ly"]
        else:
            self.px, self.py = self.dX, self.dY
            self.x0 = (self.cell % self.nx).double() * self.dX
            self.y0 = torch.div(self.cell, self.nx, rounding_mode="floor").double() * self.dY
            f["x"], f["y"] = f["x"] - self.x0, f["y"] - self.y0
        z = torch.zeros(self.nc, dtype=torch.float64, device="cuda")
        self.win = torch.stack([z] * 5)
        self.q, self.tgt = torch.stack([z] * 4), torch.stack([z] * 4)
        self.have = False
        self.drag = [torch.zeros_like(f["x"]) for _ in range(3)]
        self.pairs, self.age = None, 0

    def _cells(self):
        ix = torch.clamp(torch.floor(self.f["x"] / self.dX), 0, self.nx - 1).long()
        iy = torch.clamp(torch.floor(self.f["y"] / self.dY), 0, self.ny * self.nens - 1).long()
        return iy * self.nx + ix

    def _near(self, xa, ya, ra, xb, yb, rb, skin):
        dx, dy = xb - xa, yb - ya
        dx, dy = dx - self.px * torch.round(dx / self.px), dy - self.py * torch.round(dy / self.py)
        return dx * dx + dy * dy < (ra + rb + skin) ** 2

    def _search(self):
        f = self.f
        x, y, r = f["x"], f["y"], f["r"]
        fast = float(torch.sqrt(f["u"] ** 2 + f["v"] ** 2).max()) + 0.05 * self.dX / (self.EVERY * self.dt * 10)
        skin = 4.0 * fast * self.dt * self.EVERY
        I, J = [], []
        if self.truth:
            n, step = x.shape[0], max(1, (1 << 27) // max(1, x.shape[0]))
            for a in range(0, n, step):
                s = slice(a, min(n, a + step))
                hit = self._near(x[s, None], y[s, None], r[s, None], x[None, a:], y[None, a:], r[None, a:], skin)
                k = torch.nonzero(hit)
                k = k[k[:, 0] < k[:, 1]] + a
                I.append(k[:, 0]), J.append(k[:, 1])
        else:
            by = torch.argsort(self.cell, stable=True)
            n = torch.bincount(self.cell, minlength=self.nc)
            first = torch.cumsum(n, 0) - n
            n_sorted, cells = torch.sort(n, descending=True)
            sizes = n_sorted.cpu().numpy()
            c = 0
            while c < self.nc and sizes[c] > 1:
                w = int(sizes[c])
                e = min(self.nc, c + max(1, (1 << 26) // (w * w)))
                col = torch.arange(w, device="cuda")
                on = col[None] < n_sorted[c:e, None]
                who = by[torch.where(on, first[cells[c:e], None] + col[None], 0)]
                X, Y, Rr = x[who], y[who], torch.where(on, r[who], -1.0e30)
                hit = self._near(X[:, :, None], Y[:, :, None], Rr[:, :, None], X[:, None], Y[:, None], Rr[:, None], skin)
                hit &= on[:, :, None] & on[:, None] & (col[:, None] < col[None])
                k = torch.nonzero(hit)
                I.append(who[k[:, 0], k[:, 1]]), J.append(who[k[:, 0], k[:, 2]])
                c = e
        self.pairs = (torch.cat(I), torch.cat(J)) if I else (torch.zeros(0, dtype=torch.long, device="cuda"),) * 2

    def step(self):
        p, f, dt = self.p, self.f, self.dt
        if self.age == 0:
            self._search()
        self.age = (self.age + 1) % self.EVERY
        i, j = self.pairs
        x, y, u, v, w, r, h = (f[k] for k in ("x", "y", "u", "v", "omega", "r", "h"))
        dx, dy = x[j] - x[i], y[j] - y[i]
        dx, dy = dx - self.px * torch.round(dx / self.px), dy - self.py * torch.round(dy / self.py)
        d2 = dx * dx + dy * dy
        on = torch.nonzero((d2 > 0) & (d2 < (r[i] + r[j]) ** 2))[:, 0]
        i, j, dx, dy, d = i[on], j[on], dx[on], dy[on], torch.sqrt(d2[on])
        ri, rj = r[i], r[j]
        ex, ey, delta = dx / d, dy / d, d - (ri + rj)
        half = (d * d + ri * ri - rj * rj) / (2 * d)
        chord = torch.where(d <= (ri - rj).abs(), 2 * torch.minimum(ri, rj), 2 * torch.sqrt(torch.clamp(ri * ri - half * half, min=0)))
        k = chord * torch.minimum(h[i], h[j]) / p["h_ref"]
        du, dv = u[j] - u[i], v[j] - v[i]
        fn = torch.clamp(k * (p["E"] * delta + p["eta"] * (du * ex + dv * ey)), max=0)
        ft = k * p["G"] * (-du * ey + dv * ex - w[j] * rj - w[i] * ri)
        ft = torch.maximum(torch.minimum(ft, -p["mu"] * fn), p["mu"] * fn)
        fx, fy, tq = torch.zeros_like(x), torch.zeros_like(x), torch.zeros_like(x)
        gx, gy = fn * ex - ft * ey, fn * ey + ft * ex
        fx.index_add_(0, i, gx), fy.index_add_(0, i, gy), tq.index_add_(0, i, ri * ft)
        fx.index_add_(0, j, -gx), fy.index_add_(0, j, -gy), tq.index_add_(0, j, rj * ft)
        X, Y = (x, y) if self.truth else (self.x0 + x, self.y0 + y)
        uo, vo, curl = torch.full_like(x, p["uo_x"]), torch.full_like(x, p["uo_y"]), torch.zeros_like(x)
        for A, kx, ky, ph in np.asarray(p.get("modes", np.zeros((0, 4)))):
            kx, ky = 2 * math.pi * kx / p["Lx"], 2 * math.pi * ky / p["Ly"]
            th = kx * X + ky * Y + ph
            c, s = torch.cos(th), torch.sin(th)
            uo, vo, curl = uo - A * ky * c, vo + A * kx * c, curl - A * (kx * kx + ky * ky) * s
        for Au, Av, kx, ky, ph in np.asarray(p.get("vmodes", np.zeros((0, 5)))):
            th = kx * X + ky * Y + ph
            c, s = torch.cos(th), torch.sin(th)
            uo, vo, curl = uo + Au * c, vo + Av * c, curl - (Av * kx - Au * ky) * s
        turn = 2 * math.pi / p["wind_period"] * self.steps * dt if p["wind_period"] > 0 else 0.0
        wx = p["wind_x"] * math.cos(turn) - p["wind_y"] * math.sin(turn)
        wy = p["wind_x"] * math.sin(turn) + p["wind_y"] * math.cos(turn)
        so = torch.sqrt((uo - u) ** 2 + (vo - v) ** 2)
        sa = torch.sqrt((wx - u) ** 2 + (wy - v) ** 2)
        co, ca = p["Cd"] * p["rho_o"] * math.pi * r * r, p["Ca"] * p["rho_a"] * math.pi * r * r
        Dx, Dy = co * (uo - u) * so + ca * (wx - u) * sa, co * (vo - v) * so + ca * (wy - v) * sa
        lag = 0.5 * curl - w
        Dt = co * r * r * lag * lag.abs()
        m = p["rho_ice"] * math.pi * r * r * h
        inert = m * r * r * (0.5 if p["inertia_half"] else 1.0)
        f["x"], f["y"] = torch.remainder(x + dt * u, self.px), torch.remainder(y + dt * v, self.py)
        f["theta"] = f["theta"] + dt * w
        f["u"], f["v"], f["omega"] = u + dt * (fx + Dx) / m, v + dt * (fy + Dy) / m, w + dt * (tq + Dt) / inert
        self.drag = [Dx, Dy, Dt]
        self.steps += 1
        if self.truth or not p["couple"]:
            return
        N0, n_t = p["N0"], p["n_t"]
        at = (self.steps - 1) % N0 + 1
        if self.have and at % n_t == 0:
            k, share = at // n_t, n_t / N0
            s = self.tgt[0]
            f["r"] = r * ((1 + (s - 1) * k * share) / (1 + (s - 1) * (k - 1) * share))[self.cell]
            for name, t in (("u", 1), ("v", 2), ("omega", 3)):
                f[name] = f[name] + (self.tgt[t] * share)[self.cell]
            self.age = 0
        mo = self.moments()
        M = mo[:, 1]
        for t in (0, 1):
            self.win[t] += torch.where(M > 0, mo[:, 2 + t] / torch.clamp(M, min=1e-300), 0.0)
        for t in (2, 3, 4):
            self.win[t] += mo[:, 7 + t]
        if at == N0:
            self._coarse(mo)

    def _coarse(self, mo):
        p, A = self.p, self.dX * self.dY
        grid = lambda a: a.reshape(self.nens, self.ny, self.nx)  # noqa: E731
        if not self.have:
            self.q = torch.stack([mo[:, 1], mo[:, 2], mo[:, 3], mo[:, 5]]) / A
        V = [grid(self.win[t] / p["N0"]) for t in (0, 1)]
        S = [torch.zeros_like(V[0])] + [grid(self.win[t] / p["N0"] / A) for t in (2, 3, 4)]
        dT = p["N0"] * self.dt
        q = [grid(a).clone() for a in self.q]
        for e in range(self.nens):
            fast = max(float(V[0][e].abs().max()) / self.dX, float(V[1][e].abs().max()) / self.dY)
            n = max(1, math.ceil(dT * fast / 0.5))
            tau = dT / n
            vx, vy = V[0][e], V[1][e]
            E, W = (lambda a: torch.roll(a, -1, 1)), (lambda a: torch.roll(a, 1, 1))
            N, So = (lambda a: torch.roll(a, -1, 0)), (lambda a: torch.roll(a, 1, 0))
            for _ in range(n):
                new = []
                for k in range(4):
                    a = q[k][e]
                    mean = 0.25 * (E(a) + W(a) + N(a) + So(a))
                    if k in (0, 3):
                        flux = tau / (2 * self.dX) * (E(vx) * E(a) - W(vx) * W(a)) + tau / (2 * self.dY) * (N(vy) * N(a) - So(vy) * So(a))
                    else:
                        flux = tau * vx / (2 * self.dX) * (E(a) - W(a)) + tau * vy / (2 * self.dY) * (N(a) - So(a))
                    new.append(mean - flux + tau * S[k][e])
                for k in range(4):
                    q[k][e] = new[k]
        self.q = torch.stack([a.reshape(-1) for a in q])
        M, held = mo[:, 1], mo[:, 1] > 0
        s = torch.where(held, torch.sqrt(torch.clamp(self.q[0], min=0) * A / torch.where(held, M, 1.0)), 1.0)
        heavy, inert = s ** 2 * M, s ** 4 * mo[:, 4]
        of = lambda a, b: torch.where(b > 0, a / torch.where(b > 0, b, 1.0), 0.0)  # noqa: E731
        self.tgt = torch.stack([s, of(self.q[1] * A - s ** 2 * mo[:, 2], heavy), of(self.q[2] * A - s ** 2 * mo[:, 3], heavy),
                                of(self.q[3] * A - s ** 4 * mo[:, 5], inert)])
        self.win = torch.zeros_like(self.win)
        self.have = True

    def moments(self):
        p, f = self.p, self.f
        cell = self._cells() if self.truth else self.cell
        r, h, u, v, w = (f[k] for k in ("r", "h", "u", "v", "omega"))
        m = p["rho_ice"] * math.pi * r * r * h
        inert = m * r * r * (0.5 if p["inertia_half"] else 1.0)
        cols = [torch.ones_like(m), m, m * u, m * v, inert, inert * w, math.pi * r * r, m * u * u, m * v * v, *self.drag]
        out = torch.zeros(self.nc, 12, dtype=torch.float64, device="cuda")
        return out.index_add_(0, cell, torch.stack(cols, 1))

    def state(self):
        f = dict(self.f)
        if not self.truth:
            f["x"], f["y"] = f["x"] + self.x0, f["y"] + self.y0
        return {k: f[k] for k in FLOES}
