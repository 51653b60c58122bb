"""Flow schedules by the graph's largest weighted degree (waves up to 4, a trial wave up to 6,
pulses above): graphs at and beside both limits, every call that chooses, against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_1012_0006_gb300 import inputs as I

pytestmark = pytest.mark.gpu

FIELDS = ("flow", "cut_before", "cut_after", "wA_after", "wB_after", "corridor_n", "corridor_arcs", "accepted")


def _graph(top, scale):
    """A 48 x 40 grid with diagonals kept while no vertex's weighted degree exceeds top (scale: weight
    of an edge); one vertex has exactly top."""
    nx, ny = 48, 40
    i = np.arange(nx * ny).reshape(nx, ny)
    pairs = [(i[:, :-1], i[:, 1:]), (i[:-1], i[1:]), (i[:-1, :-1], i[1:, 1:]), (i[:-1, 1:], i[1:, :-1])]
    deg, edges = np.zeros(nx * ny, int), []
    rng = np.random.Generator(np.random.Philox(top))
    for a, b in pairs:
        e = np.stack([a.ravel(), b.ravel()], 1)
        for u, v in e[rng.permutation(len(e))]:
            if max(deg[u], deg[v]) + scale <= top:
                deg[u] += scale
                deg[v] += scale
                edges.append((u, v))
    assert deg.max() == top
    n, e = nx * ny, np.array(edges, np.int64)
    key = np.unique(np.concatenate([e[:, 0] * n + e[:, 1], e[:, 1] * n + e[:, 0]]))
    u, v = key // n, (key % n).astype(np.int32)
    xadj = np.concatenate([[0], np.cumsum(np.bincount(u, minlength=n))]).astype(np.int32)
    vw = np.ones(n, np.int32)
    coords = np.stack([np.repeat(np.arange(nx), ny), np.tile(np.arange(ny), nx)], 1).astype(np.float64)
    part = np.asarray(I.rcb(coords, vw, 6), np.int32)
    I.noise(xadj, v, vw, 6, part, 60, 3)
    return dict(n=n, nnz=len(v), xadj=xadj, adjncy=v, adjwgt=np.full(len(v), scale, np.int32), vwgt=vw, part=part, k=6,
                eps=0.1, alpha=4.0)


@pytest.mark.parametrize("top,scale", [(2, 1), (4, 1), (4, 2), (5, 1), (6, 1), (6, 3), (7, 1), (8, 2), (8, 1)])
def test_schedules_by_degree(gpu_lib, top, scale):
    import torch
    F = gpu_lib
    w = _graph(top, scale)
    g = F.DeviceGraph.from_workload(w)

    def dev():
        return torch.as_tensor(np.array(w["part"], np.int32)).cuda()

    def same(got, ref):
        for f in FIELDS:
            x, y = ((r[f] if isinstance(r, dict) else getattr(r, f)) for r in (got, ref))
            assert x == y, f

    with F.Context(0) as ctx:
        for sched in (0, 1):
            for okw in (dict(mb=1), dict(mb=0), dict(mb=1, fm_permille=50)):
                opts = F.default_options(sweep_sched=sched, **okw)
                st, pref, rref, _ = O.refine_batch(w, opts=O.options(**okw))
                part = dev()
                _, res, _ = ctx.refine_batch(g, part, 6, w["eps"], w["alpha"], opts)
                assert st == 0 and len(res) == len(rref)
                for a, b in zip(res, rref):
                    same(a, b)
                assert np.array_equal(part.cpu().numpy(), pref)
                st, pref, rref, _ = O.refine_active(w, opts=O.options(**okw), max_outer=2)
                part = dev()
                _, res, _, _ = ctx.refine_active(g, part, 6, w["eps"], w["alpha"], opts, max_outer=2)
                assert st == 0 and len(res) == len(rref)
                for a, b in zip(res, rref):
                    same(a, b)
                assert np.array_equal(part.cpu().numpy(), pref)
                pa, pb, _, _ = O.rounds(w)
                st, pref, rref = O.refine_pair(w, int(pa[0]), int(pb[0]), opts=O.options(**okw))
                part = dev()
                _, res = ctx.refine_pair(g, part, 6, int(pa[0]), int(pb[0]), w["eps"], w["alpha"], opts)
                assert st == 0
                same(res, rref)
                assert np.array_equal(part.cpu().numpy(), pref)
