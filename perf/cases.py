"""Workloads of the refinement library: what its users run, through its public calls.

A case is a dict of plain numbers and texts.  Its "call" says which entry point it takes
(pair, batch, host, active, cycle, kway, serve), its "graph" which generator of
paper_1012_0006_gb300/inputs.py makes the input, and the rest are sizes and options.
Graphs, weights, partitions and boundary noise come from the seed; the partition is
recursive coordinate bisection plus noise, as a multilevel partitioner's projected
partition would be.  Every output is whole numbers.
"""
import math

import numpy as np
import torch

from paper_1012_0006_gb300 import flowref as F, inputs as I

_KEPT = {}


def _context():
    """The stream and the context that a program keeps for all its refinements."""
    if not _KEPT:
        stream = torch.cuda.Stream()
        _KEPT.update(stream=stream, ctx=F.Context(0, stream=stream.cuda_stream))
    return _KEPT["stream"], _KEPT["ctx"]


def listed():
    return [
        # The smallest call: one plain refinement of a 4,096-vertex grid bisection; launches and waits are what it costs.
        dict(name="pair_grid2d_64", call="pair", graph="grid2d", nx=64, ny=64, swaps=200, k=2, eps=0.03, alpha=1.0,
             mb=0),
        # One block pair refined to convergence: adaptive flow iterations, alpha up to 16, on a 65,536-vertex bisection.
        dict(name="pair_rgg2d_adaptive", call="pair", graph="rgg2d", n=65536, deg=8.0, noise=20000, weights="unit", k=2,
             eps=0.03, alpha=1.0, mb=0, adaptive=1, alpha_max=16.0),
        # The widest corridor of one pair (about half the graph), most balanced cut: too large for one cluster's memory.
        dict(name="pair_rgg2d_wide_mb", call="pair", graph="rgg2d", n=65536, deg=8.0, noise=20000, weights="unit", k=2,
             eps=0.03, alpha=16.0, mb=1),
        # A small sweep as a coarse multilevel level brings it: odd n, odd k, weighted, three topological sweeps.
        dict(name="batch_rgg2d_20011_k7", call="batch", graph="rgg2d", n=20011, deg=8.0, noise=20000, weights="random",
             k=7, eps=0.03, alpha=2.0, mb=1, reps=3, results=1),
        # A mesh: the 128^3 seven-point grid in 16 blocks, one sweep, per-pair results read.
        dict(name="batch_grid3d_128_k16", call="batch", graph="grid3d", nx=128, ny=128, nz=128, noise=10000, k=16,
             eps=0.03, alpha=2.0, mb=1, results=1),
        # The large sweep: 4.2 M vertices, 50 M directed edges, 64 weighted blocks.
        dict(name="batch_rgg3d_4M_k64", call="batch", graph="rgg3d", n=4194304, deg=12.0, noise=10000,
             weights="random", k=64, eps=0.01, alpha=4.0, mb=1, results=0),
        # The same through host buffers: graph and partition uploaded, partition read back.
        dict(name="host_rgg3d_524287_k32", call="host", graph="rgg3d", n=524287, deg=12.0, noise=10000,
             weights="random", k=32, eps=0.01, alpha=4.0, mb=1),
        # A sweep with two-way FM before every flow (the 5 % rule).
        dict(name="batch_fm_rgg3d_262144_k64", call="batch", graph="rgg3d", n=262144, deg=12.0, noise=10000,
             weights="random", k=64, eps=0.01, alpha=4.0, mb=1, fm=50, results=1),
        # The strong setting: active block scheduling, FM, adaptive flows, multi-try FM after every matching.
        dict(name="active_strong_rgg3d_131071_k32", call="active", graph="rgg3d", n=131071, deg=12.0, noise=10000,
             weights="random", k=32, eps=0.03, alpha=1.0, mb=1, fm=50, adaptive=1, alpha_max=8.0, mt=10, outer=4),
        # Multilevel: one V-cycle with the given partition, a sweep on every level.
        dict(name="vcycle_rgg3d_1000003_k64", call="cycle", kind="V", graph="rgg3d", n=1000003, deg=12.0, noise=10000,
             weights="random", k=64, eps=0.01, alpha=4.0, mb=1),
        # Global k-way FM rounds from the whole boundary, until a round gains nothing (ten at most).
        dict(name="kway_rgg3d_524288_k64", call="kway", graph="rgg3d", n=524288, deg=12.0, noise=10000,
             weights="random", k=64, eps=0.01, alpha=10, init=0, rounds=10),
        # The serving loop: a burst of 24 requests on nine resident graphs of 1 K to 65 K vertices.
        dict(name="serve_24_requests", call="serve", graphs=9, max_n=65536, requests=24, inflight=32, alpha=2.0, mb=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["pair", "pair", "batch", "batch", "batch", "host", "active", "cycle", "kway", "serve"])
    if call == "pair":
        adaptive = rng.randint(0, 1)
        case = dict(call=call, k=2, eps=0.03, alpha=1.0 if adaptive else float(rng.choice([1, 2, 4, 8, 16])),
                    mb=rng.randint(0, 1), adaptive=adaptive, alpha_max=float(rng.choice([4, 8, 16])))
        if rng.random() < 0.3:
            nx, ny = _log(rng, 32, 256), _log(rng, 32, 256)
            return dict(case, graph="grid2d", nx=nx, ny=ny, swaps=max(8, 3 * ny))
        return dict(case, graph="rgg2d", n=_log(rng, 2000, 100000), deg=float(rng.choice([8, 10])), noise=20000,
                    weights=rng.choice(["unit", "random"]))
    if call == "serve":
        return dict(call=call, graphs=rng.randint(3, 9), max_n=_log(rng, 4096, 65536), requests=rng.randint(4, 32),
                    inflight=rng.choice([4, 16, 32]), alpha=2.0, mb=rng.randint(0, 1))
    n = _log(rng, 16384, {"active": 131072, "cycle": 800000, "kway": 700000, "host": 1000000}.get(call, 3000000))
    # blocks of 1 K to 64 K vertices, as the listed sweeps have
    k = min(128, max(4, _log(rng, max(4, n / 65536), max(5, n / 1024))))
    case = dict(call=call, k=k, mb=rng.randint(0, 1), eps=rng.choice([0.01, 0.03]))
    kind = rng.choice(["grid3d", "rgg2d", "rgg3d", "rgg3d"])
    if kind == "grid3d":
        s = n ** (1.0 / 3.0)
        nx, ny = int(s * rng.uniform(0.7, 1.3)), int(s * rng.uniform(0.7, 1.3))
        case.update(graph=kind, nx=nx, ny=ny, nz=max(4, n // (nx * ny)), noise=10000)
    else:
        case.update(graph=kind, n=n, deg=8.0 if kind == "rgg2d" else 12.0, noise=10000,
                    weights=rng.choice(["unit", "random"]))
    flow = dict(alpha=float(rng.choice([1, 2, 4])), reps=rng.choice([1, 1, 3]))
    if call == "batch":
        return dict(case, **flow, fm=rng.choice([0, 0, 10, 50]) if n <= 262144 else 0, results=rng.randint(0, 1))
    if call == "host":
        return dict(case, **flow)
    if call == "active":
        return dict(case, alpha=1.0, fm=rng.choice([0, 50]), adaptive=rng.randint(0, 1),
                    alpha_max=float(rng.choice([2, 8])), mt=rng.choice([0, 10]), outer=rng.choice([2, 4]))
    if call == "cycle":
        return dict(case, alpha=float(rng.choice([2, 4])), kind="V" if n > 65536 else rng.choice(["V", "W", "F"]))
    return dict(case, alpha=10, init=rng.randint(0, 1), rounds=rng.choice([1, 3, 10]))


def _workload(case, seed):
    """The seeded input: CSR arrays, weights and the partition to refine."""
    s = (I.SEED_BASE + 7919 * seed) & 0x7FFFFFFF
    g, k = case["graph"], case["k"]
    if g == "grid2d":
        return I.grid2d_halves(case["nx"], case["ny"], case["swaps"], s)
    if g == "grid3d":
        return I.grid3d_rcb(case["nx"], case["ny"], case["nz"], k, case["noise"], s)
    dim, n = (2 if g == "rgg2d" else 3), case["n"]
    if dim == 3 and case["weights"] == "random":
        return I.rgg3d_rcb(n, case["deg"], k, case["noise"], s)
    xadj, adj, coords = I.rgg(dim, n, I.rgg_radius(dim, n, case["deg"]), s)
    if case["weights"] == "random":
        vwgt, adjwgt = I.uniform_i32(n, 1, 4, s ^ 0x22), I.edge_weights(xadj, adj, 1, 10, s ^ 0x11)
    else:
        vwgt, adjwgt = np.ones(n, np.int32), np.ones(len(adj), np.int32)
    part = I.rcb(coords, vwgt, k, force_axis=0 if k == 2 else -1)
    I.noise(xadj, adj, vwgt, k, part, -case["noise"], s ^ 0x33)
    return dict(xadj=xadj, adjncy=adj, adjwgt=adjwgt, vwgt=vwgt, part=part)


def _pool(case, seed):
    """A server's graphs: 2D grids and 2D/3D random geometric graphs, 1,024 vertices up to max_n."""
    pool = []
    for i in range(case["graphs"]):
        s = (I.SEED_BASE + 104729 * seed + 31 * i) & 0x7FFFFFFF
        n = int(1024 * (case["max_n"] / 1024) ** (i / max(1, case["graphs"] - 1)))
        if i % 3 == 0:
            xadj, adj, coords = I.grid2d(math.isqrt(n), math.isqrt(n))
        else:
            dim = 2 + i % 2
            xadj, adj, coords = I.rgg(dim, n, I.rgg_radius(dim, n, 10.0), s)
        n = len(xadj) - 1
        adjwgt = np.ones(len(adj), np.int32) if i % 2 else I.edge_weights(xadj, adj, 1, 10, s ^ 0x11)
        pool.append(dict(n=n, xadj=xadj, adjncy=adj, adjwgt=adjwgt, vwgt=np.ones(n, np.int32), coords=coords, seed=s))
    return pool


def _options(case):
    return F.default_options(mb=case.get("mb", 0), mb_reps=case.get("reps", 1), adaptive=case.get("adaptive", 0),
                             max_iters=10, alpha_max=max(case.get("alpha_max", 1.0), float(case["alpha"])),
                             fm_permille=case.get("fm", 0), mt_alpha=case.get("mt", 0))


class _Serving:
    """A server with its resident graphs; closed with the state that holds it."""

    def __init__(self, case, pool):
        self.server = F.Server(0, max_inflight=case["inflight"], opts=_options(case))
        self.ids = [self.server.add_graph(g["xadj"], g["adjncy"], g["adjwgt"], g["vwgt"]) for g in pool]

    def __del__(self):
        self.server.close()


def prepare(case, seed):
    if case["call"] == "serve":
        pool = _pool(case, seed)
        rs = np.random.Generator(np.random.Philox(case["requests"]))
        requests = []
        for _ in range(case["requests"]):
            gi, k = int(rs.integers(0, len(pool))), int(rs.choice([2, 4, 8, 16]))
            requests.append((gi, I.serving_partition(pool[gi], k), k, float(rs.choice([0.01, 0.03, 0.05]))))
        return dict(case=case, serving=_Serving(case, pool), requests=requests, sizes=[g["n"] for g in pool])
    w = _workload(case, seed)
    state = dict(case=case, opts=_options(case))
    if case["call"] == "host":
        pin = lambda a: torch.as_tensor(np.ascontiguousarray(a, np.int32)).pin_memory()  # noqa: E731
        _context()
        return dict(state, arrays=[pin(w[x]) for x in ("xadj", "adjncy", "adjwgt", "vwgt")], part0=pin(w["part"]),
                    part=pin(w["part"]))
    stream, _ = _context()
    with torch.cuda.stream(stream):
        state.update(graph=F.DeviceGraph.from_workload(w), part0=torch.as_tensor(w["part"]).cuda())
        state["part"] = state["part0"].clone()
    stream.synchronize()
    return state


# What a pair's refinement found; the remaining fields of its result describe the search for it.
_FOUND = ("a", "b", "round", "flow", "cut_before", "cut_fm", "cut_after", "wA_after", "wB_after", "corridor_n",
          "corridor_arcs", "accepted", "iters", "fm_moves", "status")
_TOTALS = ("npairs", "nrounds", "accepted", "cut_before", "cut_after", "mt_gain", "mt_kept")


def _pairs(res, room):
    """The refined pairs, one row each, in a table with room for every pair there can be."""
    out = np.full((room, len(_FOUND)), -1, np.int64)
    if res:
        out[:len(res)] = [[r[f] for f in _FOUND] for r in res]
    return out


def run(state):
    case = state["case"]
    call, k = case["call"], case.get("k")
    if call == "serve":
        srv = state["serving"].server
        for tag, (gi, part, kr, eps) in enumerate(state["requests"]):
            srv.submit(state["serving"].ids[gi], part, kr, eps, case["alpha"], tag)
        out = {}
        for _ in state["requests"]:
            resp, part = srv.next(max(state["sizes"]), timeout_ms=60000)
            out[resp["tag"]] = (part[:state["sizes"][state["requests"][resp["tag"]][0]]],
                                [resp[f] for f in ("status", "npairs", "nrounds", "accepted", "cut_before",
                                                   "cut_after")])
        return [out[t][0] for t in sorted(out)] + [np.array([out[t][1] for t in sorted(out)], np.int64)]
    stream, ctx = _context()
    eps, alpha, opts, part = case["eps"], case["alpha"], state["opts"], state["part"]
    if call == "host":
        part.copy_(state["part0"])
        summ = ctx.refine_batch_host(*state["arrays"], part, k, eps, alpha, opts)
        return dict(part=part, totals=[summ[f] for f in _TOTALS])
    graph = state["graph"]
    with torch.cuda.stream(stream):
        part.copy_(state["part0"])
    if call == "pair":
        _, res = ctx.refine_pair(graph, part, k, 0, 1, eps, alpha, opts)
        return dict(part=part, pair=[getattr(res, f) for f in _FOUND if f != "round"])
    if call == "batch":
        _, res, summ = ctx.refine_batch(graph, part, k, eps, alpha, opts, results=bool(case["results"]))
        return dict(part=part, pairs=_pairs(res, k * (k - 1) // 2), totals=[summ[f] for f in _TOTALS])
    if call == "active":
        _, res, summ, outer = ctx.refine_active(graph, part, k, eps, alpha, opts, max_outer=case["outer"])
        return dict(part=part, pairs=_pairs(res, case["outer"] * k * (k - 1) // 2),
                    totals=[summ[f] for f in _TOTALS], outer=outer)
    if call == "cycle":
        _, res = ctx.cycle(graph, part, k, eps, alpha, kind=case["kind"], opts=opts)
        return dict(part=part, counts=[res[f] for f in ("coarsenings", "refinements", "depth")],
                    cuts=[res["cut_before"], res["cut_after"]])
    _, res = ctx.kway_global(graph, part, k, eps, init_mode=case["init"], alpha=case["alpha"],
                             max_rounds=case["rounds"], seed=1)
    return dict(part=part, totals=[res[f] for f in ("gain", "searches", "tried", "kept")])


def work(case):
    """Each input array read once, the partition written once; the arithmetic is on whole numbers."""
    if case["call"] == "serve":   # requests on graphs of a quarter of max_n vertices and 8 arcs a vertex, on average
        n = case["requests"] * case["max_n"] / 4
        return {"bytes": 4.0 * (4 * n + 2 * 8 * n), "flops": 0.0}
    if case["graph"] == "grid2d":
        n = case["nx"] * case["ny"]
        nnz = 4 * n - 2 * (case["nx"] + case["ny"])
    elif case["graph"] == "grid3d":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        n = nx * ny * nz
        nnz = 6 * n - 2 * (nx * ny + ny * nz + nx * nz)
    else:                         # a few per cent of the expected degree are lost at the border
        n = case["n"]
        nnz = 0.98 * case["deg"] * n
    return {"bytes": 4.0 * ((n + 1) + n + 2 * nnz + 2 * n), "flops": 0.0}


def exact(case, seed):
    """Every output is whole numbers, compared as they are."""
    return None
