"""The calls whose speed matters to a user of this library, as measurable cases.

Each kind is one public entry point over the range of sizes this repository's
workloads declare: viewpoint counts from 30 (the tiny grid) to 3000 (the
serving stream's longest tours), swarms and tour counts from one tour to the
bridge swarm's 4096, 0 to 20 obstacle boxes.

  fitness    dpso_fitness: scoring a swarm's tours on a cost matrix
  cost       dpso_cost_matrix: straight-segment edge costs of a site survey
  astar      dpso_cost_matrix_astar: edge costs by A* over the voxel grid
  two_opt    dpso_two_opt / dpso_two_opt_noalloc: polishing tours from elsewhere
  node_swap  dpso_node_swap: the node-swap exchange on such tours
  plan       dpso_plan: one solve from host arrays to host tour
  swarm      Swarm: a solve on a device cost matrix with its whole state returned
  batch      Batch: many uneven instances solved in step
  serve      Server: a burst of re-planning requests to a running server
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1706_04399_gb300 import dpso, inputs


def listed():
    return [
        # scoring a bridge swarm once: a generation's gathers on their own
        {"name": "fitness_bridge", "kind": "fitness", "shape": "bridge", "n": 1992, "count": 4096},
        # a site's edge costs before any solve, among clutter
        {"name": "cost_bridge", "kind": "cost", "shape": "bridge", "n": 1992, "m": 20},
        # the paper's own edge costs for a facade: A* over 0.5 m voxels
        {"name": "astar_facade", "kind": "astar", "shape": "facade", "n": 400, "m": 5},
        # polishing a facade swarm's worth of tours to 2-optimality
        {"name": "two_opt_facade", "kind": "two_opt", "shape": "facade", "n": 400, "count": 1024,
         "max_moves": 0, "noalloc": False},
        # an on-board loop that may not allocate polishes a few candidate tours
        {"name": "two_opt_onboard", "kind": "two_opt", "shape": "grid", "n": 157, "count": 48,
         "max_moves": 0, "noalloc": True},
        # the longest tours of the serving stream, about one per SM
        {"name": "two_opt_long", "kind": "two_opt", "shape": "grid", "n": 2999, "count": 150,
         "max_moves": 0, "noalloc": False},
        # the node-swap reading of the exchange on facade tours
        {"name": "node_swap_facade", "kind": "node_swap", "shape": "facade", "n": 400,
         "count": 512, "max_moves": 0},
        # the smallest solve: thirty viewpoints, where launches and set-up count
        {"name": "plan_tiny", "kind": "plan", "shape": "grid", "n": 30, "m": 1, "swarm": 32,
         "generations": 200},
        # the ordinary solve: a facade from host arrays to a tour
        {"name": "plan_facade", "kind": "plan", "shape": "facade", "n": 400, "m": 5,
         "swarm": 1024, "generations": 30},
        # the large solve: a bridge swarm's first generations, state checkpointed
        {"name": "swarm_bridge", "kind": "swarm", "shape": "bridge", "n": 1992, "swarm": 512,
         "generations": 2, "exchange": "two_opt", "w": 1.0},
        # several sites of uneven size planned together
        {"name": "batch_mixed", "kind": "batch", "members": 12, "n_lo": 50, "n_hi": 700,
         "swarm": 256, "generations": 4},
        # a burst of re-planning requests on a server that is already running
        {"name": "serve_burst", "kind": "serve", "requests": 10, "n_lo": 50, "n_hi": 220,
         "swarm": 256, "generations": 20},
    ]


def _log_int(rng, lo, hi):
    hi = max(lo, hi)
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["fitness", "cost", "astar", "two_opt", "two_opt", "node_swap", "plan",
                       "swarm", "batch", "serve"])
    shape = rng.choice(["grid", "random"])
    n = _log_int(rng, 30, 2999)
    if kind == "fitness":
        return {"kind": kind, "shape": shape, "n": n, "count": _log_int(rng, 1, 4096)}
    if kind == "cost":
        return {"kind": kind, "shape": shape, "n": min(n, 1992), "m": rng.randint(0, 20)}
    if kind == "astar":
        return {"kind": kind, "shape": "grid", "n": _log_int(rng, 30, 400), "m": rng.randint(0, 5)}
    if kind == "two_opt":
        # work grows about as count n^3; no more than the longest listed case
        noalloc = rng.random() < 0.3
        n = min(n, 700) if noalloc else n
        cap = min(1024.0, (40 if noalloc else 150) * (2999.0 / n) ** 3 / (80 if noalloc else 1))
        return {"kind": kind, "shape": shape, "n": n, "count": _log_int(rng, 1, max(1, int(cap))),
                "max_moves": rng.choice([0, 0, 0, 40]), "noalloc": noalloc}
    if kind == "node_swap":
        n = min(n, 999)
        cap = min(1024.0, 512 * (400.0 / n) ** 3)
        return {"kind": kind, "shape": shape, "n": n, "count": _log_int(rng, 1, max(1, int(cap))),
                "max_moves": rng.choice([0, 0, 40])}
    if kind == "plan":
        n = min(n, 400)
        swarm = _log_int(rng, 16, 1024)
        gens = min(300, max(2, int(30 * 1024 * (400.0 / n) ** 2.9 / swarm)))
        return {"kind": kind, "shape": shape, "n": n, "m": rng.randint(0, 10), "swarm": swarm,
                "generations": _log_int(rng, 1, gens)}
    if kind == "swarm":
        swarm = _log_int(rng, 16, max(16, min(1024, int(512 * (1992.0 / n) ** 2.9))))
        exchange = rng.choice(["two_opt", "two_opt", "none", "mutation_only"])
        gens = rng.randint(1, 2) if n > 700 else rng.randint(2, 12)
        return {"kind": kind, "shape": shape, "n": min(n, 1992), "swarm": swarm,
                "generations": gens, "exchange": exchange, "w": rng.choice([1.0, 1.0, 0.7])}
    if kind == "batch":
        return {"kind": kind, "members": rng.randint(2, 12), "n_lo": 50,
                "n_hi": _log_int(rng, 100, 700), "swarm": _log_int(rng, 32, 256),
                "generations": rng.randint(1, 4)}
    return {"kind": "serve", "requests": rng.randint(2, 10), "n_lo": 50,
            "n_hi": _log_int(rng, 60, 220), "swarm": _log_int(rng, 32, 256),
            "generations": rng.randint(5, 20)}


# ------------------------------------------------------------------ inputs

def _instance(shape, n, m, seed, swarm=1, iterations=1):
    if shape == "facade":
        return inputs.facade(seed)
    if shape == "bridge":
        return inputs.bridge(seed)
    if shape == "random":
        return inputs.random_instance(n, m, seed)
    # a planar grid with clutter, as the batched and serving workloads draw it
    rng = np.random.default_rng(seed)
    spacing = float(rng.uniform(0.5, 2.0))
    rows = max(1, math.isqrt(n))
    cols = -(-n // rows)
    c = rng.uniform((0.0, 0.0, -0.5), (cols * spacing, rows * spacing, 0.5), size=(m, 3))
    half = rng.uniform(0.25, 1.0, size=(m, 3)) * spacing
    return inputs.planar_grid(n, spacing, np.concatenate([c - half, c + half], axis=1),
                              "grid", swarm, iterations, seed)


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _cost_matrix(inst):
    C = torch.empty((inst.n, inst.n), dtype=torch.int32, device="cuda")
    boxes = _gpu(inst.boxes) if inst.m else None
    dpso.dpso_cost_matrix(_gpu(inst.xyz), inst.n, boxes, inst.m, dpso.default_cost_params(), C)
    return C


def _tours(n, count, seed):
    """`count` random tours: argsorts of seeded uniform draws, as uint16 bits."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    u = torch.rand((count, n), generator=g, device="cuda", dtype=torch.float64)
    return u.argsort(dim=1).to(torch.int16)


def _members(case, seed):
    """Instances with sizes evenly spaced on the logarithm of the range, in an
    order that mixes them, each with 0 to 10 boxes."""
    rng = np.random.default_rng(seed)
    count = case.get("members", case.get("requests"))
    ratio = case["n_hi"] / case["n_lo"]
    ns = [int(round(case["n_lo"] * ratio ** ((k + 0.5) / count))) for k in range(count)]
    return [_instance("grid", ns[k * 7 % count if count % 7 else k], int(rng.integers(0, 11)),
                      seed * 64 + k) for k in range(count)]


def _voxels(case, inst, voxel_m):
    """A grid over the shape's whole extent (grids at the widest spacing) and 3 m around it."""
    if case["shape"] == "facade":
        lo, hi = (0.0, -4.0, 0.0), (40.0, -2.0, 30.0)
    else:
        rows = max(1, math.isqrt(inst.n))
        lo, hi = (0.0, 0.0, 0.0), (2.0 * -(-inst.n // rows), 2.0 * rows, 0.0)
    lo, hi = np.array(lo) - 3.0, np.array(hi) + 3.0
    return lo, np.ceil((hi - lo) / voxel_m).astype(np.int32)


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "seed": seed}
    if kind in ("batch", "serve"):
        st["inst"] = _members(case, seed)
        st["params"] = dpso.default_params(swarm=case["swarm"])
        if kind == "batch":
            st["C"] = [_cost_matrix(i) for i in st["inst"]]
        else:
            st["server"] = dpso.Server(dpso.default_server_params(max_active=16))
        return st
    inst = _instance(case["shape"], case["n"], case.get("m", 5), seed)
    st["inst"] = inst
    n = inst.n
    if kind == "plan":
        st["params"] = dpso.default_params(swarm=case["swarm"])
    elif kind in ("cost", "astar"):
        st["xyz"] = _gpu(inst.xyz)
        st["boxes"] = _gpu(inst.boxes) if inst.m else None
        st["C"] = torch.empty((n, n), dtype=torch.int32, device="cuda")
        if kind == "astar":
            origin, dims = _voxels(case, inst, 0.5)
            st["ap"] = dpso.astar_params(origin, 0.5, dims, inputs.inflate_r2(0.5, 0.5))
            st["occ"] = torch.empty(int(np.prod(dims)), dtype=torch.uint8, device="cuda")
    elif kind == "swarm":
        st["C"] = _cost_matrix(inst)
        flags = dpso.FLAG_DET_INIT | dpso.FLAG_MUTATION
        if case["exchange"] != "none":
            flags |= dpso.FLAG_TWO_OPT
        st["params"] = dpso.default_params(
            swarm=case["swarm"], flags=flags, w=case["w"],
            two_opt_trigger=1 if case["exchange"] == "mutation_only" else 0)
    else:
        st["C"] = _cost_matrix(inst)
        st["tours"] = _tours(n, case["count"], seed)
        st["work"] = st["tours"].clone()
        st["cost"] = torch.empty(case["count"], dtype=torch.int64, device="cuda")
    return st


# --------------------------------------------------------------------- run

def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "fitness":
        dpso.dpso_fitness(st["C"], st["inst"].n, st["tours"], case["count"], st["cost"])
        return {"cost": st["cost"]}
    if kind == "cost":
        i = st["inst"]
        dpso.dpso_cost_matrix(st["xyz"], i.n, st["boxes"], i.m, dpso.default_cost_params(), st["C"])
        return {"C": st["C"]}
    if kind == "astar":
        i = st["inst"]
        dpso.dpso_voxel_occupancy(st["boxes"], i.m, st["ap"], st["occ"])
        dpso.dpso_cost_matrix_astar(st["xyz"], i.n, st["occ"], st["ap"], st["C"])
        return {"occ": st["occ"], "C": st["C"]}
    if kind in ("two_opt", "node_swap"):
        fn = dpso.dpso_node_swap if kind == "node_swap" else (
            dpso.dpso_two_opt_noalloc if case["noalloc"] else dpso.dpso_two_opt)
        st["work"].copy_(st["tours"])  # the call rewrites its tours in place
        pairs, moves = fn(st["C"], st["inst"].n, st["work"], case["count"], st["cost"],
                          case["max_moves"])
        return {"tours": st["work"], "cost": st["cost"], "pairs": pairs, "moves": moves}
    if kind == "plan":
        i = st["inst"]
        tour, cost = dpso.dpso_plan(i.xyz, i.boxes, i.tags, dpso.default_cost_params(),
                                    st["params"], st["seed"], case["generations"])
        return {"tour": tour, "cost": cost}
    if kind == "swarm":
        sw = dpso.Swarm(st["C"], st["inst"].n, st["inst"].tags, st["params"], st["seed"])
        sw.step(case["generations"])
        tour, cost = sw.best()
        s = sw.state()
        sw.close()
        return {"tour": tour, "cost": cost,
                **{k: s[k].view(np.int16) for k in ("X", "V", "P")},
                **{k: s[k] for k in ("F", "PF", "history")},
                "pairs": s["pairs"], "moves": s["moves"], "runs": s["runs"]}
    if kind == "batch":
        sws = [dpso.Swarm(C, i.n, i.tags, st["params"], st["seed"] + k)
               for k, (C, i) in enumerate(zip(st["C"], st["inst"]))]
        batch = dpso.Batch(sws)
        batch.step(case["generations"])
        best = [sw.best() for sw in sws]
        hist = [sw.history() for sw in sws]
        batch.close()
        for sw in sws:
            sw.close()
        return {"tours": [t for t, _ in best], "costs": np.array([c for _, c in best]),
                "history": np.stack(hist)}
    srv, cp = st["server"], dpso.default_cost_params()
    ids = [srv.submit(i.xyz, i.boxes, i.tags, cp, st["params"], st["seed"] + k,
                      case["generations"]) for k, i in enumerate(st["inst"])]
    for rid in ids:
        srv.wait(rid)
    got = [srv.poll(rid) for rid in ids]
    return {"states": np.array([g[0] for g in got]), "tours": [g[1] for g in got],
            "costs": np.array([g[2] for g in got])}


# ----------------------------------------------------------- work and oracle

def work(case):
    """Every input read once, every output written once; flops where the call
    is arithmetic on coordinates (about 25 per box test)."""
    kind = case["kind"]
    if kind in ("batch", "serve"):
        count = case.get("members", case.get("requests"))
        n = math.sqrt(case["n_lo"] * case["n_hi"])
        per = case["generations"] * case["swarm"] * n * 2 * 4
        return {"bytes": count * (4 * n * n * (2 if kind == "serve" else 1) + per), "flops": 0}
    n = case["n"]
    if kind == "fitness":
        return {"bytes": min(4 * n * n, 4 * n * case["count"]) + case["count"] * (2 * n + 8),
                "flops": 0}
    if kind == "cost":
        return {"bytes": 4 * n * n + 24 * n + 48 * case["m"],
                "flops": n * (n - 1) / 2 * (10 + 25 * case["m"])}
    if kind == "astar":
        return {"bytes": 4 * n * n + 24 * n, "flops": 0}
    if kind in ("two_opt", "node_swap"):
        return {"bytes": 4 * n * n + case["count"] * (4 * n + 8), "flops": 0}
    # a generation reads X, V, P of every particle and writes X, V
    per = case["generations"] * case["swarm"] * n * 2 * 5
    return {"bytes": 4 * n * n + per, "flops": 0}


def _exact_cost(inst):
    p = inst.xyz
    d = p[None, :, :] - p[:, None, :]
    base = np.rint(1000.0 * np.sqrt((d[..., 0] ** 2 + d[..., 1] ** 2) + d[..., 2] ** 2))
    blocked = np.zeros((inst.n, inst.n), dtype=bool)
    with np.errstate(divide="ignore", invalid="ignore"):
        for box in inst.boxes:
            tmin = np.zeros((inst.n, inst.n))
            tmax = np.ones((inst.n, inst.n))
            ok = np.ones((inst.n, inst.n), dtype=bool)
            for k in range(3):
                dk, pk = d[..., k], p[:, None, k]
                t1, t2 = (box[k] - pk) / dk, (box[3 + k] - pk) / dk
                flat = dk == 0.0
                ok &= ~(flat & ((pk < box[k]) | (pk > box[3 + k])))
                tmin = np.where(flat, tmin, np.maximum(tmin, np.minimum(t1, t2)))
                tmax = np.where(flat, tmax, np.minimum(tmax, np.maximum(t1, t2)))
            blocked |= ok & (tmin <= tmax)
    c = np.triu(base + np.where(blocked, 1e6, 0.0), 1)
    return (c + c.T).astype(np.int64)


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("cost", "fitness"):
        return None  # tours are the outcome of a search: whole numbers, compared as they are
    inst = _instance(case["shape"], case["n"], case.get("m", 5), seed)
    C = _exact_cost(inst)
    if kind == "cost":
        return {"C": C.astype(np.int32)}
    t = _tours(inst.n, case["count"], seed).cpu().numpy().astype(np.int64)
    return {"cost": C[t, np.roll(t, -1, axis=1)].sum(axis=1)}
