"""The workloads whose speed is measured: what a program that uses libecmc has it do.

Each case is one pass of such a program through the public entry points of
`paper_2004_11040_gb300` (`ecmc.System`, the C-ABI calls of the same names,
`batch.run_batched`, `serve.Server`), from the smallest call to a box of a
million disks. Kinds of pass:

  resident  a system kept on the device runs `legs` legs and is read back
  job       a system is created from host arrays, runs, is read back and freed
  sweep     a resident system runs `legs` legs along +x, then as many along +y
            (Sec. 1: the direction has to change for the method to be
            irreducible), and is read back
  batch     many resident systems of uneven size run to a liftings budget in
            persistent launches over all of them, and are read back
  serve     a stream of requests that have arrived is served to completion
  noalloc   one leg on device arrays through the entry that allocates nothing

Starts: "lattice", the seeded jittered square lattices of the benchmark (every
row of disks is a ring of its own), and "hex", a jittered triangular lattice
near melting, where a chain lifts across rows as it does in a dense fluid.
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

from paper_2004_11040_gb300 import batch, ecmc, serve, synth


def listed():
    return [
        # the smallest call: a test-sized box, where launches and copies count
        dict(name="small_256", kind="resident", start="lattice", n=256, eta=0.70, k=4, ell=0.5,
             legs=8, cells="default", graph=False),
        # one leg at a time on device arrays, inside a program that owns the heap
        dict(name="noalloc_64k", kind="noalloc", start="lattice", n=65536, eta=0.708, k=256,
             ell=1.0, legs=1, cells="default", graph=False),
        # a medium box with about sqrt(N) chains, cells aligned with the lattice
        dict(name="lattice_16k", kind="resident", start="lattice", n=16384, eta=0.708, k=128,
             ell=1.0, legs=16, cells="lattice", graph=False),
        # the benchmark's step end to end: create, ten legs, read back, free
        dict(name="lattice_1m_job", kind="job", start="lattice", n=1048576, eta=0.72, k=1024,
             ell=1.0, legs=10, cells="lattice", graph=False),
        # the same box with as many chains as the benchmark's sweep goes to
        dict(name="lattice_1m_k16384", kind="resident", start="lattice", n=1048576, eta=0.72,
             k=16384, ell=1.0, legs=20, cells="lattice", graph=False),
        # the benchmark's step in constraint-graph mode, end to end
        dict(name="graph_1m_job", kind="job", start="lattice", n=1048576, eta=0.72, k=1024,
             ell=1.0, legs=10, cells="lattice", graph=True),
        # the paper's box and chain count (N = 256^2, k = 80), production sweeps
        dict(name="hex_64k_sweep", kind="sweep", start="hex", n=65536, eta=0.70, k=80, ell=1.0,
             legs=8, cells="default", graph=False),
        # the same in constraint-graph mode, as the paper's own program finds liftings
        dict(name="hex_64k_graph_sweep", kind="sweep", start="hex", n=65536, eta=0.70, k=80,
             ell=1.0, legs=8, cells="default", graph=True),
        # a large two-dimensional box with many chains
        dict(name="hex_256k_k2048", kind="resident", start="hex", n=262144, eta=0.66, k=2048,
             ell=1.0, legs=8, cells="default", graph=False),
        # replicas of uneven size advanced together (cell scan, constraint graph)
        dict(name="batch_128", kind="batch", replicas=128, budget=50000, legs=16, cells="lattice",
             graph=False),
        dict(name="batch_128_graph", kind="batch", replicas=128, budget=50000, legs=16,
             cells="lattice", graph=True),
        # independent requests served together, results read back as they finish
        dict(name="serve_12", kind="serve", requests=12, n_max=262144, budget_max=1000000, legs=8,
             graph=False),
    ]


MOST_LIFTS = 3_000_000  # of one pass of a drawn case


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["resident", "resident", "job", "sweep", "batch", "serve", "noalloc"])
    graph = kind != "noalloc" and rng.random() < 0.35
    if kind == "batch":
        return dict(kind=kind, replicas=log_int(8, 120), budget=log_int(5000, 25000),
                    legs=rng.choice([4, 16, 64]), cells="lattice", graph=graph)
    if kind == "serve":
        return dict(kind=kind, requests=log_int(2, 11), n_max=log_int(16384, 262144),
                    budget_max=log_int(100000, 400000), legs=rng.choice([4, 8, 16]), graph=graph)
    start = "hex" if kind == "sweep" else rng.choice(["lattice", "lattice", "hex"])
    n = log_int(256, 65536 if kind == "noalloc" else 1_000_000)
    eta = round(rng.uniform(0.60, 0.72 if start == "hex" else 0.74), 4)
    k = log_int(4, max(4, min(4096, n // 32)))
    if kind == "noalloc":
        k = min(k, 192)
    ell = 1.0 if n > 4000 else round(rng.uniform(0.4, 1.0), 3)
    most = int(MOST_LIFTS / (rate(start, eta) * ell * k))
    legs = 1 if kind == "noalloc" else max(1, min(rng.choice([2, 5, 10, 20]), most // 2))
    cells = "default" if start == "hex" else rng.choice(["lattice", "lattice", "default"])
    return dict(kind=kind, start=start, n=n, eta=eta, k=k, ell=ell, legs=legs, cells=cells,
                graph=graph)


# ------------------------------------------------------------------ inputs

def hex_start(n, eta, k, seed):
    """Triangular lattice of about n disks (d = 1) in a square box at packing
    fraction eta, each disk displaced inside the circle that keeps it clear of
    its neighbours; k distinct start disks."""
    rows = max(4, 2 * int(round(math.sqrt(n * 2.0 / math.sqrt(3.0)) / 2.0)))
    cols = max(4, int(round(n / rows)))
    n = rows * cols
    box = math.sqrt(n * math.pi / (4.0 * eta))
    sx, sy = box / cols, box / rows
    least = min(sx, math.hypot(0.5 * sx, sy))  # distance of nearest sites
    reach = 0.49 * (least - 1.0)
    rng = np.random.default_rng(seed)
    r, phi = reach * np.sqrt(rng.random(n)), 2.0 * math.pi * rng.random(n)
    i = np.arange(n) % cols
    j = np.arange(n) // cols
    x = np.mod((i + 0.25 + 0.5 * (j % 2)) * sx + r * np.cos(phi), box)
    y = np.mod((j + 0.5) * sy + r * np.sin(phi), box)
    x[x >= box] = 0.0
    y[y >= box] = 0.0
    return synth.Start(x=x, y=y, active=rng.choice(n, k, replace=False).astype(np.int32), box=box,
                       d=1.0, m=0, seed=seed)


def make_start(case, seed):
    if case["start"] == "hex":
        return hex_start(case["n"], case["eta"], case["k"], seed)
    m = synth.lattice_m_for(case["n"])
    return synth.lattice_start(m, case["eta"], min(case["k"], m * m), seed)


def pinned(a):
    t = torch.from_numpy(np.ascontiguousarray(a))
    return t.pin_memory() if torch.cuda.is_available() else t


def cells_of(case, start):
    return start.m if case["cells"] == "lattice" else 0


class Server(serve.Server):
    """The library's server, closed when the program drops it (as a System is)."""

    def __del__(self):
        try:
            self.close()
        except Exception:
            pass


def out_buffers(n, k):
    return {"x": pinned(np.zeros(n)), "y": pinned(np.zeros(n)), "t": pinned(np.zeros(n)),
            "active": pinned(np.zeros(k, dtype=np.int32))}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        # sizes and densities are the case's (the batched recipe), positions the seed's
        reps = [batch.Replica(synth.lattice_start(r.start.m, r.eta, r.start.k, seed * 7919 + q),
                              r.ell, r.eta)
                for q, r in enumerate(batch.make_replicas(case["replicas"], case["replicas"]))]
        systems = batch.create(reps, case["cells"], graph=case["graph"])
        out = out_buffers(sum(s.n for s in systems), sum(s.k for s in systems))
        views, at, ak = [], 0, 0
        for s in systems:
            views.append([out[f][at:at + s.n] for f in ("x", "y", "t")] +
                         [out["active"][ak:ak + s.k]])
            at, ak = at + s.n, ak + s.k
        return {"case": case, "systems": systems, "out": out, "views": views}
    if kind == "serve":
        reqs = serve.make_requests(case["requests"], case["requests"], rate=0.0,
                                   n_range=(4096, case["n_max"]),
                                   budget_range=(2e4, case["budget_max"]))
        for q, r in enumerate(reqs):
            r.seed = seed * 100003 + q
        serve.prepare(reqs)
        server = Server(64 << 30, slice_legs=case["legs"], keep_results=True, graph=case["graph"])
        return {"case": case, "requests": reqs, "server": server}
    s = make_start(case, seed)
    if kind == "noalloc":
        return {"case": case, "start": s, "x": torch.from_numpy(s.x).cuda(),
                "y": torch.from_numpy(s.y).cuda(), "active": torch.from_numpy(s.active).cuda(),
                "t": torch.zeros(s.n, dtype=torch.float64, device="cuda")}
    st = {"case": case, "out": out_buffers(s.n, s.k)}
    if kind == "job":
        flags = ecmc.ECMC_GRAPH if case["graph"] else 0
        st["params"] = ecmc.ecmc_params(s.n, s.box, s.d, case["ell"], s.k, cells_of(case, s),
                                        flags, 0, 0, 1, 0)
        st["in"] = pinned(s.x), pinned(s.y), pinned(s.active)
        return st
    st["system"] = ecmc.System(s.x, s.y, s.active, s.box, case["ell"],
                               cells_per_side=cells_of(case, s), graph=case["graph"])
    return st


# -------------------------------------------------------------------- pass

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "resident":
        system, out = state["system"], state["out"]
        flags, _ = system.run(case["legs"])
        ecmc.ecmc_positions(system.ctx, out["x"], out["y"], out["t"], out["active"])
        return {**out, "flags": flags}
    if kind == "sweep":
        system, out = state["system"], state["out"]
        fx, _ = system.run(case["legs"])
        system.set_direction(1)
        fy, _ = system.run(case["legs"])
        ecmc.ecmc_positions(system.ctx, out["x"], out["y"], out["t"], out["active"])
        system.set_direction(0)
        return {**out, "flags": fx, "flags_y": fy}
    if kind == "job":
        out = state["out"]
        flags = np.zeros(case["legs"], dtype=np.uint8)
        ctx = ecmc.ecmc_create(state["params"], *state["in"])
        ecmc.ecmc_run_to_breakpoint(ctx, case["legs"], 0, flags)
        ecmc.ecmc_positions(ctx, out["x"], out["y"], out["t"], out["active"])
        ecmc.ecmc_destroy(ctx)
        return {**out, "flags": flags}
    if kind == "batch":
        lifts, _, _ = batch.run_batched(state["systems"], case["budget"], case["legs"])
        for s, v in zip(state["systems"], state["views"]):
            ecmc.ecmc_positions(s.ctx, *v)
        return {**state["out"], "liftings": lifts}
    if kind == "serve":
        reqs = [dataclasses.replace(r) for r in state["requests"]]
        state["server"].serve(reqs)
        return {"results": [list(r.result) for r in reqs],
                "liftings": np.asarray([r.liftings for r in reqs])}
    s = state["start"]
    flag, lifts = ecmc.ecmc_leg_noalloc(s.n, s.box, s.d, case["ell"], s.k, cells_of(case, s),
                                        state["x"], state["y"], state["active"], state["t"])
    return {"x": state["x"], "active": state["active"], "t": state["t"], "flags": flag,
            "liftings": lifts}


# -------------------------------------------------------------------- work

LIFT_BYTES = 104  # three neighbours' x, y, t read; x_i, t_i, t_j and two owner words written
LIFT_FLOPS = 15   # three times of flight (two subtractions, a square root's input), three updates


def rate(start, eta):
    """Liftings per unit of chain length: one per gap of a lattice row; from
    the pressure (the rate is (Z - 1) over the mean contact distance) for a
    dense two-dimensional box."""
    if start == "lattice":
        return 1.0 / (math.sqrt(math.pi / (4.0 * eta)) - 0.9999)
    z = 1.0 / (1.0 - 1.9682 * eta + 0.9716 * eta * eta)  # Santos, Lopez de Haro & Yuste 1995
    return (z - 1.0) * 4.0 / math.pi


def work(case):
    kind = case["kind"]
    if kind == "batch":
        lifts = case["replicas"] * case["budget"]
        n = case["replicas"] * 15500  # mean of the log-uniform sizes
        return {"bytes": lifts * LIFT_BYTES + 24 * n, "flops": lifts * LIFT_FLOPS}
    if kind == "serve":
        lifts = case["requests"] * (case["budget_max"] - 2e4) / math.log(case["budget_max"] / 2e4)
        n = case["requests"] * (case["n_max"] - 4096) / math.log(case["n_max"] / 4096)
        return {"bytes": lifts * LIFT_BYTES + 40 * n, "flops": lifts * LIFT_FLOPS}
    lifts = case["k"] * case["ell"] * case["legs"] * rate(case["start"], case["eta"])
    moves = {"resident": 24, "job": 40, "sweep": 24, "noalloc": 32}[kind]
    lifts *= 2 if kind == "sweep" else 1
    return {"bytes": lifts * LIFT_BYTES + moves * case["n"], "flops": lifts * LIFT_FLOPS}


# ------------------------------------------------------------------- exact

def global_leg(x, y, active, box, d, ell):
    """One leg of the global-time process (the event of least time first, ties
    by chain) in numpy: new x, leg-relative local times, new active disks."""
    n, k = len(x), len(active)
    order = np.argsort(y, kind="stable")
    ys = y[order]
    x, t = x.copy(), np.zeros(n)
    act = np.array(active, dtype=np.int64)
    taken = np.zeros(n, dtype=bool)  # active or stalled
    taken[act] = True
    left, now = np.full(k, ell), np.zeros(k)

    def next_event(c):
        i = act[c]
        lo, hi = y[i] - d, y[i] + d
        parts = [order[np.searchsorted(ys, lo):np.searchsorted(ys, hi, "right")]]
        if lo < 0.0:
            parts.append(order[np.searchsorted(ys, lo + box):])
        if hi >= box:
            parts.append(order[:np.searchsorted(ys, hi - box, "right")])
        j = np.concatenate(parts)
        j = j[~taken[j]]
        dy = np.abs(y[j] - y[i])
        dy = np.minimum(dy, box - dy)
        ok = dy < d
        j, dy = j[ok], dy[ok]
        if not len(j):
            return left[c], -1
        dx = x[j] - x[i]
        dx[dx < 0.0] += box
        tau = np.maximum(dx - np.sqrt(d * d - dy * dy), 0.0)
        tau[now[c] + tau < t[j]] += box  # passed before j came there: a lap away
        best = tau.min()
        return (best, int(j[tau == best].min())) if best < left[c] else (left[c], -1)

    tau, target = np.zeros(k), np.zeros(k, dtype=np.int64)
    for c in range(k):
        tau[c], target[c] = next_event(c)
    running = np.ones(k, dtype=bool)
    while running.any():
        c = int(np.argmin(np.where(running, now + tau, np.inf)))
        i, j = act[c], target[c]
        t_new = now[c] + tau[c]
        x[i] = x[i] + tau[c]
        if x[i] >= box:
            x[i] -= box
        t[i] = now[c] = t_new
        left[c] = left[c] - tau[c]
        if j < 0:
            running[c] = False
            continue
        t[j] = t_new
        taken[i], taken[j] = False, True
        act[c] = j
        dy = np.abs(y[act] - y[i])
        again = running & ((np.minimum(dy, box - dy) < d) | (target == j))
        again[c] = True
        for q in np.flatnonzero(again):
            tau[q], target[q] = next_event(q)
    return x, t, act.astype(np.int32)


def exact(case, seed):
    if case["kind"] in ("batch", "serve"):
        return None
    lifts = case["k"] * case["ell"] * case["legs"] * rate(case["start"], case["eta"])
    lifts *= 2 if case["kind"] == "sweep" else 1
    if lifts * (1.0 + 0.002 * math.sqrt(case["n"])) > 60000:
        return None
    s = make_start(case, seed)
    x, y, act, t = s.x, s.y, s.active, np.zeros(s.n)
    for _ in range(case["legs"]):
        x, t, act = global_leg(x, y, act, s.box, s.d, case["ell"])
    if case["kind"] == "sweep":
        for _ in range(case["legs"]):
            y, t, act = global_leg(y, x, act, s.box, s.d, case["ell"])
    if case["kind"] == "noalloc":
        return {"x": x, "active": act, "t": t, "flags": None, "liftings": None}
    got = {"x": x, "y": y, "t": t, "active": act, "flags": None}
    return {**got, "flags_y": None} if case["kind"] == "sweep" else got
