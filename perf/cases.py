"""The work a user of this library has it do, as cases that can be timed.

Every case goes through the public entry points of ``paper_2001_06231_gb300``
with the systems of ``workloads.py``; sizes are those of the benchmark, the
served mix and the tests, and odd ones in between.  A case is a dict of plain
values; ``prepare`` makes what a program holds before the call (inputs on the
GPU, the abstraction handle, the schedule it keeps), ``run`` is one call.
"""
import math

import numpy as np
import torch

import paper_2001_06231_gb300 as bf
from paper_2001_06231_gb300 import workloads as wl

INF = float("inf")
DEV = "cuda"


def listed():
    return [
        # The smallest solve: the double integrator on 64 x 64 cells at tau = 0.3
        # (the non-degenerate parity size).  A planner that replans on a small
        # grid; launches and latency are all there is.
        {"name": "di_64x64", "kind": "solve", "system": "di", "n0": 64, "n1": 64, "tuned": False},
        # An odd two-dimensional grid: lines not a multiple of anything.
        {"name": "di_301x205", "kind": "solve", "system": "di", "n0": 301, "n1": 205, "tuned": False},
        # The unicycle of the served mix, solved on a resident abstraction with
        # the schedule the library picks by itself.
        {"name": "unicycle_100x100x32", "kind": "solve", "system": "unicycle", "n0": 100, "n1": 100, "n2": 32,
         "tuned": False},
        # The unicycle of the benchmark after bf_tune: one plant, many solves.
        {"name": "unicycle_200x200x64_tuned", "kind": "solve", "system": "unicycle", "n0": 200, "n1": 200, "n2": 64,
         "tuned": True},
        # The fire model at a ragged size, default schedule.
        {"name": "fire_61x57x24x6", "kind": "solve", "system": "fire", "n0": 61, "n1": 57, "n2": 24, "n3": 6,
         "tuned": False},
        # The benchmark's fire model, tuned: the largest single solve.
        {"name": "fire_100x100x36x8_tuned", "kind": "solve", "system": "fire", "n0": 100, "n1": 100, "n2": 36, "n3": 8,
         "tuned": True},
        # Second stage of the fire-fighting mission: a running cost that depends
        # on the successor (a class of cells) and a terminal value from stage 1.
        {"name": "mission_60x60x24x6", "kind": "mission", "system": "fire", "n0": 60, "n1": 60, "n2": 24, "n3": 6},
        # Memory regulation: a third of the inputs' boxes stored, the rest
        # regenerated, with a frontier cache.
        {"name": "hybrid_60x60x24x6", "kind": "hybrid", "system": "fire", "n0": 60, "n1": 60, "n2": 24, "n3": 6,
         "stored": 5, "cache": 100000},
        # Many plants at once: uneven unicycle instances in one batched call.
        {"name": "batch_16_unicycles", "kind": "batch", "count": 16, "scale": 2.5},
        # The server under load: requests over resident small, unicycle and fire
        # systems, pinned host buffers in and out.
        {"name": "served_15", "kind": "served", "count": 15},
        # A system solved once, from its equations to the controller: build the
        # abstraction, solve, free.
        {"name": "build_200x200x64", "kind": "build", "system": "unicycle", "n0": 200, "n1": 200, "n2": 64},
        # Boxes from the caller's own reachability tool, different from cell to
        # cell, imported and solved.
        {"name": "import_97x61x23", "kind": "import", "n0": 97, "n1": 61, "n2": 23, "inputs": 7},
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    k = rng.choice(["di", "unicycle", "unicycle", "fire", "fire", "mission", "hybrid", "batch", "served", "build",
                    "import"])
    tuned = rng.random() < 0.4
    if k == "di":
        return {"kind": "solve", "system": "di", "n0": _log(rng, 32, 400), "n1": _log(rng, 32, 400), "tuned": tuned}
    if k == "unicycle":
        return {"kind": "solve", "system": "unicycle", "n0": _log(rng, 50, 200), "n1": _log(rng, 50, 200),
                "n2": _log(rng, 16, 64), "tuned": tuned}
    if k == "fire":
        return {"kind": "solve", "system": "fire", "n0": _log(rng, 40, 100), "n1": _log(rng, 40, 100),
                "n2": _log(rng, 18, 36), "n3": _log(rng, 4, 8), "tuned": tuned}
    if k == "mission":
        return {"kind": "mission", "system": "fire", "n0": _log(rng, 40, 80), "n1": _log(rng, 40, 80),
                "n2": _log(rng, 18, 36), "n3": _log(rng, 4, 8)}
    if k == "hybrid":
        return {"kind": "hybrid", "system": "fire", "n0": _log(rng, 40, 64), "n1": _log(rng, 40, 64),
                "n2": _log(rng, 18, 26), "n3": _log(rng, 4, 7), "stored": rng.randrange(0, 14),
                "cache": rng.choice([0, _log(rng, 5000, 200000)])}
    if k == "batch":
        return {"kind": "batch", "count": rng.randrange(3, 17), "scale": rng.uniform(1.2, 2.5)}
    if k == "served":
        return {"kind": "served", "count": rng.randrange(4, 16)}
    if k == "build":
        s = rng.choice(["unicycle", "fire"])
        if s == "unicycle":
            return {"kind": "build", "system": s, "n0": _log(rng, 50, 200), "n1": _log(rng, 50, 200),
                    "n2": _log(rng, 16, 64)}
        return {"kind": "build", "system": s, "n0": _log(rng, 40, 80), "n1": _log(rng, 40, 80),
                "n2": _log(rng, 18, 36), "n3": _log(rng, 4, 8)}
    return {"kind": "import", "n0": _log(rng, 20, 120), "n1": _log(rng, 20, 100), "n2": _log(rng, 5, 40),
            "inputs": rng.randrange(3, 12)}


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _fire_target():
    return ((50.0, 250.0), (50.0, 150.0), (-math.radians(30), math.radians(30)), (10.0, 15.0))


def _workload(case, seed):
    """The host workload of a single-system case: another seed moves the target,
    the obstacles or no-fly boxes, the fires and the costs."""
    rng = np.random.default_rng(seed)
    s = case["system"]
    if s == "di":
        w = wl.di2d(n=(case["n0"], case["n1"]), tau=0.3)
        cx, cy = rng.uniform(-3.5, 0.0), rng.uniform(-1.0, 1.0)
        w.target = wl.box_contains_cells(w.grid, [(cx - 0.6, cx + 0.6), (cy - 0.6, cy + 0.6)]).astype(np.uint8)
        w.target &= 1 - w.avoid
        w.G = w.G * rng.uniform(0.5, 2.0)
        return w
    if s == "unicycle":
        tx, ty = rng.uniform(1.0, 8.0, size=2)
        return wl.unicycle3d(n=(case["n0"], case["n1"], case["n2"]), seed=seed, target_xy=((tx, tx + 1.0), (ty, ty + 1.0)),
                             n_obstacles=int(rng.integers(20, 41)), cost_c=float(rng.uniform(0.05, 1.0)))
    # cells of 10 m as in the benchmark's fire model, whatever the grid's size
    n = (case["n0"], case["n1"], case["n2"], case["n3"])
    return wl.fire4d(n=n, seed=seed, target=_fire_target(), tau=2.0, extent=10.0 * max(n[0], n[1]))


def _import_arrays(case, seed):
    """Boxes int16 [C][U][2][3] that differ from cell to cell (a drift per input
    plus one cell of noise), costs, target and avoid cells; torch on the GPU."""
    n = (case["n0"], case["n1"], case["n2"])
    U, C = case["inputs"], n[0] * n[1] * n[2]
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    c = torch.arange(C, device=DEV)
    k = [c % n[0], (c // n[0]) % n[1], c // (n[0] * n[1])]
    boxes = torch.zeros((C, U, 2, 3), dtype=torch.int16, device=DEV)
    for u in range(U):
        ok = torch.rand(C, generator=g, device=DEV) >= 0.03
        lo, hi = [], []
        for d in range(3):
            drift = int(round(2.0 * math.cos(2.0 * math.pi * (u + 0.3 * d) / U + 1.5 * d)))
            l = k[d] + drift + torch.randint(-1, 2, (C,), generator=g, device=DEV)
            w = torch.randint(0, 2, (C,), generator=g, device=DEV)
            if d == 2:                                   # the last dim wraps
                l = l % n[2]
            else:
                ok &= (l >= 0) & (l + w <= n[d] - 1)
            lo.append(l)
            hi.append(l + w)
        for d in range(3):
            boxes[:, u, 0, d] = torch.where(ok, lo[d], 0).to(torch.int16)
            boxes[:, u, 1, d] = torch.where(ok, hi[d], 0).to(torch.int16)
        boxes[~ok, u, 0, 0] = bf.BLOCKED
    G = 0.125 + 0.25 * torch.randint(0, 6, (C, U), generator=g, device=DEV).to(torch.float64)
    target = (torch.rand(C, generator=g, device=DEV) < 0.004).to(torch.uint8)
    avoid = (torch.rand(C, generator=g, device=DEV) < 0.05).to(torch.uint8)
    grid = bf.make_grid(n, [0.0] * 3, [float(x) for x in n], [False, False, True])
    return grid, boxes, G, target, avoid


def _device(w):
    return {"G": torch.from_numpy(w.G).to(DEV), "target": torch.from_numpy(w.target).to(DEV),
            "avoid": torch.from_numpy(w.avoid).to(DEV)}


def _outputs(C):
    return (torch.empty(C, dtype=torch.float64, device=DEV), torch.empty(C, dtype=torch.uint8, device=DEV))


def _batch_sizes(case):
    """Uneven grids, log-uniform in scale; they belong to the case, not to the seed."""
    rng = np.random.default_rng(case["count"])
    s = np.exp(rng.uniform(0.0, math.log(case["scale"]), size=case["count"]))
    return [(int(round(50 * x)), int(round(50 * x)), int(round(16 * x))) for x in s]


def _batch_workloads(case, seed):
    rng = np.random.default_rng(seed)
    return [_workload({"system": "unicycle", "n0": n[0], "n1": n[1], "n2": n[2]}, int(rng.integers(0, 2**31 - 1)))
            for n in _batch_sizes(case)]


def _served_payloads(case, seed):
    """Requests over three resident systems (a small double integrator, a
    unicycle, a fire model), each with its own target or fire map."""
    rng = np.random.default_rng(seed)
    out = []
    for i in range(case["count"]):
        s = int(rng.integers(0, 2**31 - 1))
        c = ({"system": "di", "n0": 64, "n1": 64}, {"system": "unicycle", "n0": 100, "n1": 100, "n2": 32},
             {"system": "fire", "n0": 60, "n1": 60, "n2": 24, "n3": 6})[i % 3]
        out.append((i % 3, _workload(c, s)))
    return out


def _system(w):
    return (w.kind, w.params, w.substeps, w.grid, w.inputs, w.tau)


def _mission_inputs(w):
    """Stage costs of the mission: tau + phi^2, and -5 tau for successors over
    the fire at drop speed."""
    g2 = w.tau + np.asarray(w.inputs)[:, 0] ** 2
    G = np.ascontiguousarray(np.broadcast_to(g2, (w.ncells, w.ninputs)))
    Gc = np.full((w.ncells, w.ninputs), -5.0 * w.tau)
    cls = wl.fire4d_fire_cells(w, 0.3, (12.0, 16.5))
    return G, Gc, cls


def prepare(case, seed):
    kind = case["kind"]
    st = {"kind": kind}
    if kind == "batch":
        ws = _batch_workloads(case, seed)
        st["A"] = [bf.abs_build_workload(w) for w in ws]
        ins = [_device(w) for w in ws]
        st["G"], st["target"], st["avoid"] = ([i[k] for i in ins] for k in ("G", "target", "avoid"))
        outs = [_outputs(w.ncells) for w in ws]
        st["V"], st["mu"] = [o[0] for o in outs], [o[1] for o in outs]
        return st
    if kind == "served":
        pay = _served_payloads(case, seed)
        st["server"] = bf.Server(hbm_budget=8 << 30, max_active=64, passes_per_step=8)
        # one request per system builds the resident abstractions
        for k, w in pay[:3]:
            st["server"].poll(st["server"].submit(w.G, target=w.target, avoid=w.avoid, system=_system(w)))
        st["requests"] = [(_system(w), torch.from_numpy(w.G).pin_memory(), torch.from_numpy(w.target).pin_memory(),
                           torch.from_numpy(w.avoid).pin_memory(),
                           torch.empty(w.ncells, dtype=torch.float64).pin_memory(),
                           torch.empty(w.ncells, dtype=torch.uint8).pin_memory()) for _, w in pay]
        return st
    if kind == "import":
        st["grid"], st["boxes"], st["G"], st["target"], st["avoid"] = _import_arrays(case, seed)
        st["V"], st["mu"] = _outputs(case["n0"] * case["n1"] * case["n2"])
        return st
    w = _workload(case, seed)
    st.update(_device(w))
    st["V"], st["mu"] = _outputs(w.ncells)
    if kind == "build":
        st["w"] = w
    elif kind == "hybrid":
        st["A"] = bf.abs_build_workload(w, box_budget=8 * w.ncells * case["stored"])
        st["cache"] = case["cache"]
    elif kind == "mission":
        st["A"] = bf.abs_build_workload(w)
        G2, Gc, cls = _mission_inputs(w)
        # stage 1 (to the landing box) is the terminal value of stage 2
        G1 = torch.from_numpy(G2).to(DEV)
        r1 = bf.bf_solve(st["A"], G1, target=st["target"], avoid=st["avoid"], V=torch.empty_like(st["V"]),
                         mu=torch.empty_like(st["mu"]))
        st["G"], st["G_class"] = G1, torch.from_numpy(Gc).to(DEV)
        st["terminal"], st["cls"] = r1["V"], torch.from_numpy(cls).to(DEV)
    else:
        st["A"] = bf.abs_build_workload(w)
        if case["tuned"]:
            bf.bf_tune(st["A"], st["G"], target=st["target"], avoid=st["avoid"])
    return st


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------

def _result(r):
    return {"V": r["V"], "mu": r["mu"], "iters": r["iters"], "status": r["status"]}


def _results(rs):
    return {"V": [r["V"] for r in rs], "mu": [r["mu"] for r in rs], "iters": np.array([r["iters"] for r in rs]),
            "status": np.array([r["status"] for r in rs])}


def run(st):
    kind = st["kind"]
    if kind == "solve":
        return _result(bf.bf_solve(st["A"], st["G"], target=st["target"], avoid=st["avoid"], V=st["V"], mu=st["mu"]))
    if kind == "mission":
        return _result(bf.bf_solve(st["A"], st["G"], terminal=st["terminal"], avoid=st["avoid"], succ_class=st["cls"],
                                   G_class=st["G_class"], V=st["V"], mu=st["mu"]))
    if kind == "hybrid":
        return _result(bf.bf_solve(st["A"], st["G"], target=st["target"], avoid=st["avoid"], V=st["V"], mu=st["mu"],
                                   frontier_cache=st["cache"]))
    if kind == "batch":
        rs = bf.bf_solve_batch(st["A"], st["G"], targets=st["target"], avoids=st["avoid"], Vs=st["V"], mus=st["mu"])
        return _results(rs)
    if kind == "served":
        srv = st["server"]
        ids = [srv.submit(G, target=tg, avoid=av, system=s, borrow=True, V=V, mu=mu)
               for s, G, tg, av, V, mu in st["requests"]]
        return _results([srv.poll(i) for i in ids])
    if kind == "build":
        A = bf.abs_build_workload(st["w"])
    else:
        A = bf.abs_from_boxes(st["grid"], st["boxes"])
    r = _result(bf.bf_solve(A, st["G"], target=st["target"], avoid=st["avoid"], V=st["V"], mu=st["mu"]))
    A.close()
    return r


# --------------------------------------------------------------------------
# work
# --------------------------------------------------------------------------

def _solve_work(C, U, extra=0):
    """Costs, target and avoid read once, V and mu written once; one addition
    per (cell, input) pair at least."""
    return {"bytes": C * (8 * U + 2 + 9) + extra, "flops": C * U}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        return _solve_work(sum(a * b * c for a, b, c in _batch_sizes(case)), 10)
    if kind == "served":
        c = case["count"]
        per = [_solve_work(64 * 64, 5), _solve_work(100 * 100 * 32, 10), _solve_work(60 * 60 * 24 * 6, 15)]
        tot = {"bytes": 0, "flops": 0}
        for i in range(c):
            for k in tot:
                tot[k] += per[i % 3][k]
        return tot
    C = case["n0"] * case["n1"] * case.get("n2", 1) * case.get("n3", 1)
    if kind == "import":
        return _solve_work(C, case["inputs"], 12 * C * case["inputs"])
    U = {"di": 5, "unicycle": 10, "fire": 15}[case["system"]]
    if kind == "mission":
        return _solve_work(C, U, 8 * C * U + 8 * C)
    return _solve_work(C, U)


# --------------------------------------------------------------------------
# the value function in plain torch
# --------------------------------------------------------------------------

def _flow_boxes(w, dev):
    """Per input the first cell and the widths of every cell's box, and which
    pairs stay on the grid: the flow of the system in FP64, as in the paper
    (corner images of the linear system; RK4 centre and growth bound else)."""
    g = w.grid
    n, D = g.n, len(g.n)
    eta = [(g.hi[d] - g.lo[d]) / n[d] for d in range(D)]
    c = torch.arange(g.ncells, device=dev)
    k, r = [], c
    for d in range(D):
        k.append((r % n[d]).to(torch.float64))
        r = r // n[d]
    tau = w.tau
    for u in np.asarray(w.inputs):
        u = [float(x) for x in u]
        if D == 2:
            ends = []
            for q in range(4):
                x0 = g.lo[0] + (k[0] + (q & 1)) * eta[0]
                x1 = g.lo[1] + (k[1] + (q >> 1)) * eta[1]
                ends.append((x0 + tau * x1 + 0.5 * tau * tau * u[0], x1 + tau * u[0]))
            a = [torch.stack([e[d] for e in ends]).amin(0) for d in range(2)]
            b = [torch.stack([e[d] for e in ends]).amax(0) for d in range(2)]
        else:
            p = [float(x) for x in w.params]
            x = [g.lo[d] + (k[d] + 0.5) * eta[d] for d in range(D)]
            rad = [0.5 * e for e in eta]
            if D == 3:
                def f(s):
                    return [u[0] * torch.cos(s[2]), u[0] * torch.sin(s[2]), u[1]]

                def gr(s):
                    return [p[0] + abs(u[0]) * s[2], p[0] + abs(u[0]) * s[2], p[0]]
            else:
                def f(s):
                    return [s[3] * torch.cos(s[2]) + p[0], s[3] * torch.sin(s[2]), p[1] / s[3] * math.tan(u[0]), u[1]]

                def gr(s):
                    m = p[3] * s[2] + s[3]
                    return [p[4] + m, p[4] + m, p[4] + p[1] * math.tan(abs(u[0])) / (p[2] * p[2]) * s[3], p[4]]
            h = tau / w.substeps

            def rk4(fun, s):
                k1 = fun(s)
                k2 = fun([s[i] + 0.5 * h * k1[i] for i in range(D)])
                k3 = fun([s[i] + 0.5 * h * k2[i] for i in range(D)])
                k4 = fun([s[i] + h * k3[i] for i in range(D)])
                return [s[i] + h / 6.0 * (k1[i] + 2.0 * k2[i] + 2.0 * k3[i] + k4[i]) for i in range(D)]
            for _ in range(w.substeps):
                x, rad = rk4(f, x), rk4(gr, rad)
            a = [x[d] - rad[d] for d in range(D)]
            b = [x[d] + rad[d] for d in range(D)]
        lo, wid, ok = [], [], torch.ones(g.ncells, dtype=torch.bool, device=dev)
        for d in range(D):
            l = torch.floor((a[d] - g.lo[d]) / eta[d]).to(torch.int64)
            e = torch.floor((b[d] - g.lo[d]) / eta[d]).to(torch.int64)
            if g.periodic[d]:
                wid.append((e - l + 1).clamp(max=n[d]))
                lo.append(l % n[d])
            else:
                ok &= (l >= 0) & (e <= n[d] - 1)
                lo.append(l)
                wid.append(e - l + 1)
        yield lo, wid, ok


def _value(n, periodic, boxes, G, terminal, avoid, dev):
    """Greatest fixed point below the terminal cost, by whole sweeps."""
    D, C = len(n), int(np.prod(n))
    stride = [int(np.prod(n[:d])) for d in range(D)]
    V = torch.where(avoid, torch.full_like(terminal, INF), terminal)
    plans = []
    for u, (lo, wid, ok) in enumerate(boxes):
        sel = torch.nonzero(ok & ~avoid).flatten()
        if not sel.numel():
            continue
        dims = []
        for d in range(D):
            l, wd = lo[d][sel], wid[d][sel]
            steps = []
            for o in range(int(wd.max())):
                i = l + torch.clamp(wd - 1, max=o)
                if periodic[d]:
                    i = i % n[d]
                steps.append((i * stride[d]).to(torch.int32))
            dims.append(steps)
        plans.append((sel, dims, G[sel, u]))

    def box_max(dims, d, base, m):
        for s in dims[d]:
            i = s if base is None else base + s
            if d == 0:
                x = V[i]
                m = x if m is None else torch.maximum(m, x, out=m)
            else:
                m = box_max(dims, d - 1, i, m)
        return m
    for _ in range(C):
        W = V.clone()
        for sel, dims, g in plans:
            m = box_max(dims, D - 1, None, None)
            W[sel] = torch.minimum(W[sel], g + m)
        if torch.equal(W, V):
            break
        V = W
    return V


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "served", "mission", "hybrid"):
        return None
    C = case["n0"] * case["n1"] * case.get("n2", 1) * case.get("n3", 1)
    if C > (100_000 if case.get("system") == "fire" else 600_000):   # the fire model's boxes hold many cells
        return None
    dev = DEV if torch.cuda.is_available() else "cpu"
    if kind == "import":
        grid, boxes, G, target, avoid = _import_arrays(case, seed)
        n, periodic = [case["n0"], case["n1"], case["n2"]], [False, False, True]
        b = boxes.to(torch.int64)
        it = (([b[:, u, 0, d] for d in range(3)], [b[:, u, 1, d] - b[:, u, 0, d] + 1 for d in range(3)],
               b[:, u, 0, 0] != bf.BLOCKED) for u in range(case["inputs"]))
    else:
        w = _workload(case, seed)
        n, periodic = w.grid.n, w.grid.periodic
        it = _flow_boxes(w, dev)
        G, target, avoid = (torch.from_numpy(x).to(dev) for x in (w.G, w.target, w.avoid))
    terminal = torch.where(target != 0, 0.0, INF).to(torch.float64)
    return {"V": _value(n, periodic, it, G, terminal, avoid != 0, dev), "mu": None, "iters": None, "status": None}
