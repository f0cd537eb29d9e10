"""Measured cases of the shallow-water lattice Boltzmann library: what its users run.

A case is one job through the public entry points.  A run sets the initial state, advances it
and reads the result back; a batch does the same for many grids at once; a gradient
differentiates a run with respect to its initial depth.  Handles (``Simulation``, ``Batch``)
are made in ``prepare`` and kept, as a program that runs many jobs keeps them.

``exact`` restates the D1Q3Q2 and D2Q5Q4Q4 schemes in plain torch at 64 bits.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_1401_0427_gb300 import adjoint, lbm_sw

DEVICE = "cuda"
G = 1.0
S = 1.8
# relaxation rates of the 13 moments, ten of them distinct (the conserved ones are ignored)
MRT_RATES = [0.0, 1.1, 1.2, 1.3, 1.4, 0.0, 1.5, 1.6, 1.7, 0.0, 1.75, 1.65, 0.9]
P, W, O, I = lbm_sw.PERIODIC, lbm_sw.WALL, lbm_sw.OUTFLOW, lbm_sw.INFLOW
# sides in the order x-, x+, y-, y+
SIDES = {
    "periodic": (P, P, P, P),
    "basin": (W, W, W, W),
    "channel": (I, O, W, W),
    "reflection": (I, W, P, P),
    "open": (O, O, O, O),
}


def listed():
    return [
        # the paper's section 2 shock tube in the size of the benchmark: host arrays in, host
        # arrays out, the smallest job; latency counts
        {"name": "tube_1000_f64", "kind": "tube", "nx": 1000, "precision": "f64", "sides": "basin", "steps": 500},
        # the paper's forward-facing step on its finest mesh (section 4), in double precision
        # as the experiments run it: a small grid, solid cells, many steps
        {"name": "step_480x120_f64", "kind": "grid", "nx": 480, "ny": 120, "precision": "f64", "sides": "channel",
         "collision": "bgk", "solid": "step", "steps": 600, "every": 0, "out": "fields"},
        # a run to a steady state that checks totals and the smallest depth every few steps
        # and reads them on the host (odd sizes)
        {"name": "watch_701x401_f64", "kind": "grid", "nx": 701, "ny": 401, "precision": "f64", "sides": "basin",
         "collision": "bgk", "solid": "none", "steps": 100, "every": 10, "out": "fields"},
        # shock reflection from a wall: the 512 x 512 workload of the benchmark, half its steps
        {"name": "reflection_512_f32", "kind": "grid", "nx": 512, "ny": 512, "precision": "f32", "sides": "reflection",
         "collision": "bgk", "solid": "none", "steps": 1000, "every": 0, "out": "fields"},
        # double precision on a grid that does not fit L2
        {"name": "dam_1536_f64", "kind": "grid", "nx": 1536, "ny": 1536, "precision": "f64", "sides": "periodic",
         "collision": "bgk", "solid": "none", "steps": 60, "every": 0, "out": "fields"},
        # a closed basin of odd width and ragged height, checkpointed at the end
        {"name": "basin_2501x1803_f32", "kind": "grid", "nx": 2501, "ny": 1803, "precision": "f32", "sides": "basin",
         "collision": "bgk", "solid": "none", "steps": 120, "every": 0, "out": "state"},
        # a channel with a relaxation rate per moment
        {"name": "channel_mrt_2048x1024_f32", "kind": "grid", "nx": 2048, "ny": 1024, "precision": "f32",
         "sides": "channel", "collision": "mrt", "solid": "none", "steps": 120, "every": 0, "out": "state"},
        # a flow among islands: solid blocks scattered over a large grid
        {"name": "islands_3000x2000_f32", "kind": "grid", "nx": 3000, "ny": 2000, "precision": "f32",
         "sides": "periodic", "collision": "bgk", "solid": "islands", "steps": 60, "every": 0, "out": "state"},
        # a middle-sized periodic run
        {"name": "dam_1024_f32", "kind": "grid", "nx": 1024, "ny": 1024, "precision": "f32", "sides": "periodic",
         "collision": "bgk", "solid": "none", "steps": 200, "every": 0, "out": "state"},
        # the benchmark's circular dam break
        {"name": "dam_4096_f32", "kind": "grid", "nx": 4096, "ny": 4096, "precision": "f32", "sides": "periodic",
         "collision": "bgk", "solid": "none", "steps": 120, "every": 0, "out": "fields"},
        # an ensemble of uneven grids advanced together
        {"name": "ensemble_64_f32", "kind": "batch", "count": 64, "low": 64, "high": 1024, "precision": "f32",
         "sides": "periodic", "steps": 120},
        # one gradient of the inverse problem: recorded run, loss, discrete adjoint
        {"name": "gradient_1024_f32", "kind": "gradient", "nx": 1024, "ny": 1024, "precision": "f32",
         "sides": "periodic", "steps": 200},
    ]


def _log(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def draw(rng):
    kind = rng.choice(["tube", "grid", "grid", "grid", "grid", "batch", "gradient"])
    precision = rng.choice(["f32", "f32", "f64"])
    if kind == "tube":
        return {"kind": "tube", "nx": _log(rng, 80, 16000), "precision": rng.choice(["f32", "f64"]),
                "sides": rng.choice(["basin", "periodic", "open"]), "steps": rng.randrange(100, 1000)}
    if kind == "batch":
        low = _log(rng, 32, 200)
        return {"kind": "batch", "count": _log(rng, 4, 64), "low": low, "high": rng.randrange(low + 50, 1025),
                "precision": "f32", "sides": rng.choice(["periodic", "basin"]), "steps": rng.randrange(20, 120)}
    if kind == "gradient":
        return {"kind": "gradient", "nx": _log(rng, 64, 1024), "ny": _log(rng, 64, 1024), "precision": "f32",
                "sides": rng.choice(["periodic", "periodic", "basin"]), "steps": rng.randrange(20, 200)}
    solid = rng.choice(["none", "none", "islands", "step"])
    sides = "channel" if solid == "step" else rng.choice(["periodic", "periodic", "basin", "channel", "reflection"])
    collision = rng.choice(["bgk", "bgk", "mrt"]) if solid == "none" else "bgk"
    # cells times steps stay below the largest listed run; double precision runs at a tenth of the rate
    top = 4096 * 4096 * 60 // (25 if precision == "f64" else 1)
    if precision == "f32" and (collision == "mrt" or solid != "none"):
        top //= 4
    nx, ny = _log(rng, 96, 4096 if precision == "f32" else 2048), _log(rng, 64, 4096 if precision == "f32" else 2048)
    steps = max(1, min(rng.randrange(10, 1000), top // (nx * ny)))
    return {"kind": "grid", "nx": nx, "ny": ny, "precision": precision, "sides": sides, "collision": collision,
            "solid": solid, "steps": steps, "every": max(1, steps // 6) if precision == "f64" and rng.random() < 0.5 else 0,
            "out": rng.choice(["fields", "state"])}


# ------------------------------------------------------------------------------ inputs
def _generator(seed):
    return torch.Generator(device=DEVICE).manual_seed(int(seed))


def _uniform(gen, *shape, low=0.0, high=1.0):
    return low + (high - low) * torch.rand(*shape, generator=gen, device=DEVICE, dtype=torch.float64)


def _host_rng(seed):
    return np.random.default_rng(int(seed))


def _square(nx, ny):
    n = max(nx, ny)
    x = (torch.arange(nx, device=DEVICE, dtype=torch.float64) + 0.5) / n
    y = (torch.arange(ny, device=DEVICE, dtype=torch.float64) + 0.5) / n
    return x[None, :], y[:, None]


def _dam(nx, ny, rng, gen):
    """A column of deep water somewhere near the middle, at rest, with a perturbation of 1e-3."""
    x, y = _square(nx, ny)
    n = max(nx, ny)
    cx, cy = (rng.uniform(0.4, 0.6) * s / n for s in (nx, ny))
    r = rng.uniform(0.15, 0.25) * min(nx, ny) / n
    h = torch.where((x - cx) ** 2 + (y - cy) ** 2 < r * r, 2.0, 1.0).to(torch.float64)
    return h + _uniform(gen, ny, nx, low=-1e-3, high=1e-3)


def _bumps(nx, ny, rng):
    """Eight smooth bumps on water of depth 1 (periodic distance)."""
    x, y = ((torch.arange(m, device=DEVICE, dtype=torch.float64) + 0.5) / m for m in (nx, ny))
    h = torch.ones(ny, nx, device=DEVICE, dtype=torch.float64)
    for _ in range(8):
        a, s, cx, cy = rng.uniform(0.05, 0.3), rng.uniform(0.03, 0.1), rng.random(), rng.random()
        dx, dy = (torch.minimum((v - c).abs(), 1.0 - (v - c).abs()) for v, c in ((x, cx), (y, cy)))
        h = h + a * torch.exp(-(dy[:, None] ** 2 + dx[None, :] ** 2) / (2.0 * s * s))
    return h


def _solid(case, rng):
    nx, ny = case["nx"], case["ny"]
    mask = np.zeros((ny, nx), dtype=np.uint8)
    if case["solid"] == "step":
        # a block 0.2 high from x = 0.6 to the exit, in units of the channel's height (kept
        # inside short channels)
        mask[: max(1, round(0.2 * ny)), min(round(0.6 * ny), nx // 2):] = 1
    elif case["solid"] == "islands":
        side = max(2, min(nx, ny) // 64)
        for _ in range(48):
            x, y = int(rng.integers(0, nx - side)), int(rng.integers(0, ny - side))
            mask[y:y + side, x:x + int(rng.integers(side // 2 + 1, side + 1))] = 1
    return mask


def _grid_problem(case, seed):
    """(parameters, initial state, solid mask) of a run, all from the seed."""
    rng, gen = _host_rng(seed), _generator(seed)
    nx, ny = case["nx"], case["ny"]
    lam, inflow = 8.0, None
    if case["solid"] == "step":
        lam, froude = 80.0, rng.uniform(2.8, 3.2)
        h = 1.0 + _uniform(gen, ny, nx, low=-1e-3, high=1e-3)
        hu, hv = froude * h, torch.zeros_like(h)
        inflow = (1.0, froude, 0.0)
    elif case["sides"] == "reflection":
        left = rng.uniform(1.6, 2.2)
        u = (left - 1.0) * math.sqrt(G * (left + 1.0) / (2.0 * left))
        behind = (torch.arange(nx, device=DEVICE) < nx // 2).expand(ny, nx)
        # the shock runs into water with bumps on it, so the flow behind it is not planar
        h = torch.where(behind, left, _bumps(nx, ny, rng))
        hu, hv = torch.where(behind, left * u, 0.0).to(torch.float64), torch.zeros_like(h)
        inflow = (left, left * u, 0.0)
    else:
        h = _dam(nx, ny, rng, gen)
        hu, hv = torch.zeros_like(h), torch.zeros_like(h)
        if case["sides"] == "channel":
            hu = hu + 0.2
            inflow = (1.0, 0.2, 0.0)
    state = [t.contiguous() for t in (h, hu, hv)]
    return {"lam": lam, "a": 0.05, "inflow": inflow}, state, _solid(case, rng)


def _tube_problem(case, seed):
    rng = _host_rng(seed)
    nx = case["nx"]
    x = (np.arange(nx) + 0.5) / nx
    h = np.where(x < rng.uniform(0.4, 0.6), rng.uniform(1.5, 2.5), 1.0) + rng.uniform(-1e-3, 1e-3, nx)
    return h, np.zeros(nx)


def _batch_problem(case, seed):
    # the instances' sizes belong to the ensemble, not to the seed
    sizes = [(int(v), int(v)) for v in _host_rng(case["count"]).integers(case["low"], case["high"] + 1, case["count"])]
    gen, states = _generator(seed), []
    rng = _host_rng(seed)
    for nx, ny in sizes:
        h = _dam(nx, ny, rng, gen)
        states.append([h, torch.zeros_like(h), torch.zeros_like(h)])
    return sizes, states


def _gradient_problem(case, seed):
    rng = _host_rng(seed)
    truth, guess = (_bumps(case["nx"], case["ny"], rng) for _ in range(2))
    return guess.to(torch.float32), truth.to(torch.float32)


def _precision(case):
    return lbm_sw.FP64 if case["precision"] == "f64" else lbm_sw.FP32


def _dtype(case):
    return torch.float64 if case["precision"] == "f64" else torch.float32


def _stream():
    return torch.cuda.current_stream().cuda_stream


# ------------------------------------------------------------------------------ jobs
def prepare(case, seed):
    kind = case["kind"]
    if kind == "tube":
        sim = lbm_sw.Simulation(case["nx"], 1, dim=1, precision=_precision(case), a=0.15, s=S,
                                bc=SIDES[case["sides"]][:2], stream=_stream())
        return {"case": case, "sim": sim, "in": _tube_problem(case, seed)}
    if kind == "batch":
        sizes, states = _batch_problem(case, seed)
        batch = lbm_sw.Batch(sizes, precision=_precision(case), s=S, bc=SIDES[case["sides"]], stream=_stream())
        out = [torch.empty(13, ny, nx, device=DEVICE, dtype=_dtype(case)) for nx, ny in sizes]
        return {"case": case, "batch": batch, "in": states, "out": out}
    if kind == "gradient":
        sim = lbm_sw.Simulation(case["nx"], case["ny"], precision=_precision(case), s=S, bc=SIDES[case["sides"]],
                                stream=_stream())
        h0, seen = _gradient_problem(case, seed)
        return {"case": case, "sim": sim, "h0": h0.requires_grad_(True), "seen": seen}
    par, state, solid = _grid_problem(case, seed)
    sim = lbm_sw.Simulation(case["nx"], case["ny"], precision=_precision(case), lam=par["lam"], s=S, a=par["a"],
                            bc=SIDES[case["sides"]], inflow=[par["inflow"]] * 4 if par["inflow"] else None,
                            stream=_stream())
    if case["collision"] == "mrt":
        sim.set_relaxation(MRT_RATES)
    if case["solid"] != "none":
        sim.set_obstacle(torch.from_numpy(solid).to(DEVICE))
    if case["out"] == "fields":
        out = [torch.empty_like(state[0]) for _ in range(3)]
    else:
        out = torch.empty(13, case["ny"], case["nx"], device=DEVICE, dtype=_dtype(case))
    return {"case": case, "sim": sim, "in": state, "out": out}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "tube":
        sim = state["sim"]
        sim.set_state(*state["in"])
        sim.step(case["steps"])
        h, q = sim.moments()
        return {"h": h, "q": q}
    if kind == "batch":
        batch = state["batch"]
        for i, w in enumerate(state["in"]):
            batch.set_state(i, *w)
        batch.step(case["steps"])
        for i, out in enumerate(state["out"]):
            lbm_sw.lbm_sw_batch_get_populations(batch.handle, i, out.data_ptr(), True)
        return state["out"]
    if kind == "gradient":
        h0 = state["h0"]
        h0.grad = None
        # the model's parameter is in single precision, as torch programs keep them
        end = adjoint.run(h0.double(), state["sim"], case["steps"]).to(h0.dtype)
        loss = 0.5 * ((end - state["seen"]) ** 2).sum()
        loss.backward()
        return {"end": end.detach(), "gradient": h0.grad}
    sim = state["sim"]
    sim.set_state(*state["in"])
    totals, every, left = [], case["every"], case["steps"]
    while every and left >= every:
        sim.step(every)
        left -= every
        totals.append(sim.diagnostics()[:4])
    sim.step(left)
    if case["out"] == "state":
        sim.populations_into(state["out"])
        result = {"state": state["out"]}
    else:
        sim.moments_into(*state["out"])
        # fields of a single precision run are kept in single precision
        result = {n: t.to(_dtype(case)) for n, t in zip(("h", "hu", "hv"), state["out"])}
    if totals:
        result["totals"] = np.array(totals)
    return result


def work(case):
    """Bytes of the arrays that go in and come out; operations of the steps (a fused
    multiply-add is two)."""
    size = 8 if case["precision"] == "f64" else 4
    if case["kind"] == "tube":
        return {"bytes": case["nx"] * 32.0, "flops": 33.0 * case["nx"] * case["steps"]}
    if case["kind"] == "batch":
        cells = sum(nx * ny for nx, ny in _batch_sizes(case))
        return {"bytes": cells * (24.0 + 13 * size), "flops": 73.0 * cells * case["steps"]}
    cells = case["nx"] * case["ny"]
    if case["kind"] == "gradient":
        # forward step, and its transposed Jacobian at the moments of each step
        return {"bytes": cells * (8.0 + 4.0 + 4.0), "flops": (73.0 + 110.0) * cells * case["steps"]}
    out = 13.0 * size if case["out"] == "state" else 3.0 * size
    checks = case["steps"] // case["every"] if case["every"] else 0
    per_step = 73.0 if case["collision"] == "bgk" else 128.0
    return {"bytes": cells * (24.0 + out), "flops": cells * (per_step * case["steps"] + 13.0 * checks)}


def _batch_sizes(case):
    return [(int(v), int(v)) for v in _host_rng(case["count"]).integers(case["low"], case["high"] + 1, case["count"])]


# ------------------------------------------------------------------------------ 64 bits
# Populations of a cell: f0, f+x, f+y, f-x, f-y of the depth, then four of each discharge.
_DIRECTION = [0, 1, 2, 3, 4, 1, 2, 3, 4, 1, 2, 3, 4]


def _equilibrium(h, hu, hv, lam, a):
    u, v = hu / h, hv / h
    f0 = a * (0.5 * h - (u * u + v * v) / (4.0 * G))
    r, c, p = 0.25 * (h - f0), 0.5 / lam, 0.5 * G * h * h
    xx, yy, xy = c * (hu * u + p), c * (hv * v + p), c * hu * v
    return [f0, r + c * hu, r + c * hv, r - c * hu, r - c * hv,
            0.25 * hu + xx, 0.25 * hu + xy, 0.25 * hu - xx, 0.25 * hu - xy,
            0.25 * hv + xy, 0.25 * hv + yy, 0.25 * hv - xy, 0.25 * hv - yy]


def _moments(f):
    return sum(f[1:5], f[0]), sum(f[6:9], f[5]), sum(f[10:13], f[9])


def _collide(f, lam, a, rates):
    e = _equilibrium(*_moments(f), lam, a)
    if rates is None:
        return [x + S * (y - x) for x, y in zip(f, e)]
    d = [y - x for x, y in zip(f, e)]
    jx, jy = rates[1] * (d[1] - d[3]), rates[2] * (d[2] - d[4])
    eps = rates[3] * (d[1] + d[2] + d[3] + d[4] - 4.0 * d[0]) / 5.0
    xx = rates[4] * (d[1] - d[2] + d[3] - d[4])
    out = [f[0] - eps, f[1] + 0.25 * (eps + xx) + 0.5 * jx, f[2] + 0.25 * (eps - xx) + 0.5 * jy,
           f[3] + 0.25 * (eps + xx) - 0.5 * jx, f[4] + 0.25 * (eps - xx) - 0.5 * jy]
    for base, (ra, rb, rx) in ((5, rates[6:9]), (9, rates[10:13])):
        g = d[base:base + 4]
        ja, jb, x = ra * (g[0] - g[2]), rb * (g[1] - g[3]), rx * (g[0] - g[1] + g[2] - g[3])
        out += [f[base] + 0.25 * x + 0.5 * ja, f[base + 1] - 0.25 * x + 0.5 * jb,
                f[base + 2] + 0.25 * x - 0.5 * ja, f[base + 3] - 0.25 * x - 0.5 * jb]
    return out


def _stream_in(f, bc, inflow, near):
    """Populations arriving at each cell; `near[d]`: where the cell that direction d comes
    from is solid."""
    out = [f[0]]
    for p in range(1, 13):
        d = _DIRECTION[p]
        partner = p + 2 if d < 3 else p - 2
        along = 1 if d in (1, 3) else 0
        normal = 5 <= p <= 8 if along else p >= 9
        side = {1: 0, 3: 1, 2: 2, 4: 3}[d]
        n = f[p].shape[along]
        first = d < 3  # comes from the lower neighbour
        edge, body = f[p].narrow(along, 0 if first else n - 1, 1), f[p].narrow(along, 0 if first else 1, n - 1)
        if bc[side] == P:
            edge = f[p].narrow(along, n - 1 if first else 0, 1)
        elif bc[side] == W:
            edge = f[partner].narrow(along, 0 if first else n - 1, 1)
            edge = -edge if normal else edge
        elif bc[side] == I:
            edge = inflow[p].expand_as(edge)
        g = torch.cat([edge, body] if first else [body, edge], dim=along)
        if near is not None:
            g = torch.where(near[d], -f[partner] if normal else f[partner], g)
        out.append(g)
    return out


def _steps2d(f, steps, lam, a, bc, rates=None, inflow=None, solid=None):
    if inflow is not None:
        inflow = _equilibrium(*(torch.full((1, 1), v, device=DEVICE, dtype=torch.float64) for v in inflow), lam, a)
    near = None
    if solid is not None and bool(solid.any()):
        near = {}
        for d, (axis, shift) in {1: (1, 1), 2: (0, 1), 3: (1, -1), 4: (0, -1)}.items():
            m = torch.roll(solid, shift, dims=axis)
            if bc[{1: 0, 3: 1, 2: 2, 4: 3}[d]] != P:
                m.select(axis, 0 if shift > 0 else -1).fill_(False)
            near[d] = m & ~solid
    for _ in range(steps):
        g = _collide(_stream_in(f, bc, inflow, near), lam, a, rates)
        f = g if near is None else [torch.where(solid, x, y) for x, y in zip(f, g)]
    return f


def _steps1d(h, q, steps, bc):
    lam, a = 8.0, 0.15
    c = 0.5 / lam

    def equilibrium(h, q):
        f0 = a * (0.5 * h - (q / h) ** 2 / (4.0 * G))
        half, flux = 0.5 * (h - f0), c * (q * q / h + 0.5 * G * h * h)
        return [f0, half + c * q, half - c * q, 0.5 * q + flux, 0.5 * q - flux]

    f = equilibrium(h, q)
    for _ in range(steps):
        g = [f[0]]
        for p in (1, 2, 3, 4):
            first, partner = p in (1, 3), {1: 2, 2: 1, 3: 4, 4: 3}[p]
            rule = bc[0] if first else bc[1]
            at = slice(0, 1) if first else slice(-1, None)
            if rule == P:
                edge = f[p][-1:] if first else f[p][:1]
            elif rule == W:
                edge = -f[partner][at] if p > 2 else f[partner][at]
            else:
                edge = f[p][at]
            g.append(torch.cat([edge, f[p][:-1]] if first else [f[p][1:], edge]))
        e = equilibrium(g[0] + g[1] + g[2], g[3] + g[4])
        f = [x + S * (y - x) for x, y in zip(g, e)]
    return f[0] + f[1] + f[2], f[3] + f[4]


def exact(case, seed):
    kind = case["kind"]
    if kind == "gradient":
        return _exact_gradient(case, seed)
    with torch.no_grad():
        if kind == "tube":
            h, q = _steps1d(*(torch.from_numpy(v).to(DEVICE) for v in _tube_problem(case, seed)), case["steps"],
                            SIDES[case["sides"]][:2])
            return {"h": h, "q": q}
        if kind == "batch":
            lam, a, bc = 8.0, 0.05, SIDES[case["sides"]]
            return [torch.stack(_steps2d(_equilibrium(*w, lam, a), case["steps"], lam, a, bc))
                    for w in _batch_problem(case, seed)[1]]
        par, w, solid = _grid_problem(case, seed)
        lam, a, bc = par["lam"], par["a"], SIDES[case["sides"]]
        rates = MRT_RATES if case["collision"] == "mrt" else None
        solid = torch.from_numpy(solid).to(DEVICE).bool()
        f, totals, every, left = _equilibrium(*w, lam, a), [], case["every"], case["steps"]
        while every and left >= every:
            f = _steps2d(f, every, lam, a, bc, rates, par["inflow"], solid)
            left -= every
            m = _moments(f)
            totals.append([float(t.sum()) for t in m] + [float(m[0].min())])
        f = _steps2d(f, left, lam, a, bc, rates, par["inflow"], solid)
        result = {"state": torch.stack(f)} if case["out"] == "state" else dict(zip(("h", "hu", "hv"), _moments(f)))
        if totals:
            result["totals"] = np.array(totals)
        return result


def _exact_gradient(case, seed):
    from torch.utils.checkpoint import checkpoint

    lam, a, bc = 8.0, 0.05, SIDES[case["sides"]]
    guess, seen = (t.double() for t in _gradient_problem(case, seed))
    guess.requires_grad_(True)
    f = _equilibrium(guess, torch.zeros_like(guess), torch.zeros_like(guess), lam, a)
    left, part = case["steps"], max(1, math.isqrt(case["steps"]))
    while left > 0:
        n = min(part, left)
        f = checkpoint(lambda *g, n=n: tuple(_steps2d(list(g), n, lam, a, bc)), *f, use_reentrant=False)
        left -= n
    end = _moments(list(f))[0]
    loss = 0.5 * ((end - seen) ** 2).sum()
    (gradient,) = torch.autograd.grad(loss, guess)
    return {"end": end.detach(), "gradient": gradient}
