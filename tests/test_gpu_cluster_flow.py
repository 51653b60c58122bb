"""The cluster max flow, the queue kernel's single rounds and the FM search where their code
branches: rows of one, two and many strides, networks whose arcs mostly cross CTAs, weights
above 15 bits, waves, clusters that a network outgrows, arena bounds between the workspaces,
cluster sizes that change from call to call, FM stacks longer than their shared-memory ring.
Everything is whole numbers: equal to the oracle's."""
import numpy as np
import pytest

import oracle as O
from paper_1012_0006_gb300 import inputs as I
from tests.hub_graph import hub_workload

pytestmark = pytest.mark.gpu

FIELDS = ("flow", "cut_before", "cut_after", "wA_after", "wB_after", "corridor_n", "corridor_arcs", "accepted",
          "iters", "cut_fm", "fm_moves")


@pytest.fixture(scope="module")
def F(gpu_lib):
    return gpu_lib


@pytest.fixture(scope="module")
def ctx(F):
    c = F.Context(0)
    yield c
    c.close()


def _dev(F, w):
    import torch
    return F.DeviceGraph.from_workload(w), torch.as_tensor(np.array(w["part"], np.int32)).cuda()


def _same(got, ref):
    for f in FIELDS:
        assert got[f] == ref[f] if isinstance(got, dict) else getattr(got, f) == getattr(ref, f), f


def _pair(F, ctx, w, a=0, b=1, dev=None, **okw):
    st, pref, rref = O.refine_pair(w, a, b, opts=O.options(**okw))
    assert st == 0
    g, part = _dev(F, w)
    _, res = ctx.refine_pair(g, part, w["k"], a, b, w["eps"], w["alpha"], F.default_options(**okw, **(dev or {})))
    _same(res, rref)
    assert np.array_equal(part.cpu().numpy(), pref)
    return res


def _batch(F, ctx, w, dev=None, **okw):
    st, pref, rref, _ = O.refine_batch(w, opts=O.options(**okw))
    assert st == 0
    g, part = _dev(F, w)
    _, res, _ = ctx.refine_batch(g, part, w["k"], w["eps"], w["alpha"], F.default_options(**okw, **(dev or {})))
    assert len(res) == len(rref)
    for rg, rc in zip(res, rref):
        _same(rg, rc)
    assert np.array_equal(part.cpu().numpy(), pref)


def _active(F, ctx, w, dev=None, **okw):
    st, pref, rref, _ = O.refine_active(w, opts=O.options(**okw), max_outer=2)
    assert st == 0
    g, part = _dev(F, w)
    _, res, _, _ = ctx.refine_active(g, part, w["k"], w["eps"], w["alpha"], F.default_options(**okw, **(dev or {})),
                                     max_outer=2)
    assert len(res) == len(rref)
    for rg, rc in zip(res, rref):
        _same(rg, rc)
    assert np.array_equal(part.cpu().numpy(), pref)


def _random_regular(n, deg, scale=1):
    """A random graph without locality: most arcs of its network join two CTAs."""
    rs = np.random.Generator(np.random.Philox(n * 100 + deg))
    u = np.repeat(np.arange(n, dtype=np.int64), deg // 2)
    v = rs.integers(0, n, len(u))
    u, v = u[u != v], v[u != v]
    key = np.unique(np.concatenate([u * n + v, v * n + u]))
    u, v = key // n, (key % n).astype(np.int32)
    xadj = np.concatenate([[0], np.cumsum(np.bincount(u, minlength=n))]).astype(np.int32)
    wt = (1 + (np.minimum(u, v) * 31 + np.maximum(u, v) * 7) % 9).astype(np.int32) * scale
    part = (np.arange(n) >= n // 2).astype(np.int32)
    return dict(n=n, nnz=len(v), xadj=xadj, adjncy=v, adjwgt=wt, vwgt=np.ones(n, np.int32), part=part, k=2, eps=0.1,
                alpha=4.0, mb=0)


@pytest.mark.parametrize("ctas", [4, 16])
@pytest.mark.parametrize("deg_lo,deg_hi", [(15, 17), (31, 34), (60, 70), (500, 900)])
def test_rows_of_every_length(F, ctx, deg_lo, deg_hi, ctas):
    w = dict(hub_workload(11 + deg_lo, n=2500, hubs=10, deg_lo=deg_lo, deg_hi=deg_hi, k=4), alpha=8.0)
    _batch(F, ctx, w, dict(cluster_ctas=ctas), mb=1)
    _batch(F, ctx, w, dict(cluster_ctas=ctas, sweep_sched=1))


@pytest.mark.parametrize("scale", [1, 3000, 5000])
@pytest.mark.parametrize("n,deg", [(600, 4), (957, 4), (960, 6), (963, 8), (2000, 12), (5000, 20)])
def test_networks_that_cross_ctas(F, ctx, n, deg, scale):
    w = _random_regular(n, deg, scale)
    for dev in (dict(cluster_ctas=4), dict(cluster_ctas=16), dict(sweep_sched=1)):
        _pair(F, ctx, w, dev=dev)


@pytest.mark.parametrize("nx,k,alpha", [(96, 16, 4.0), (128, 24, 8.0)])
def test_waves_in_a_sweep(F, ctx, nx, k, alpha):
    xadj, adj, coords = I.grid2d(nx, nx)
    vwgt = np.ones(nx * nx, np.int32)
    part = I.rcb(coords, vwgt, k)
    I.noise(xadj, adj, vwgt, k, part, nx * 4, 5)
    w = dict(n=nx * nx, nnz=len(adj), xadj=xadj, adjncy=adj, adjwgt=np.ones(len(adj), np.int32), vwgt=vwgt, part=part,
             k=k, eps=0.03, alpha=alpha)
    for sched in (0, 1, 2):
        _batch(F, ctx, w, dict(flow_sched=sched), mb=1)


@pytest.mark.parametrize("fm", [0, 50])
@pytest.mark.parametrize("dev", [{}, dict(sweep_sched=1), dict(cluster_ctas=4), dict(cluster_ctas=16)], ids=str)
def test_rounds_on_the_queue_kernel(F, ctx, dev, fm):
    w = dict(I.grid3d_rcb(40, 40, 40, k=4, alpha=16.0), mb=1)   # its networks outgrow four CTAs
    pa, pb, _, _ = O.rounds(w)
    _pair(F, ctx, w, int(pa[0]), int(pb[0]), dev, mb=1, fm_permille=fm)
    w["alpha"] = 1.0
    okw = dict(mb=1, adaptive=1, max_iters=6, alpha_max=16.0, fm_permille=fm)
    _pair(F, ctx, w, int(pa[0]), int(pb[0]), dev, **okw)
    _active(F, ctx, w, dev, **okw)


@pytest.mark.parametrize("call", ["pair", "active", "batch"])
def test_arena_bounds_between_the_workspaces(F, call):
    w = dict(I.grid2d_halves(128, 128, swaps=500, alpha=4.0), mb=1)
    w["part"] = I.rcb(I.grid2d(128, 128)[2], w["vwgt"], 4)
    I.noise(w["xadj"], w["adjncy"], w["vwgt"], 4, w["part"], 300, 3)
    w["k"] = 4
    okw = dict(mb=1)
    if call == "pair":
        st, pref, _ = O.refine_pair(w, 0, 1, opts=O.options(**okw))
    elif call == "batch":
        st, pref, _, _ = O.refine_batch(w, opts=O.options(**okw))
    else:
        st, pref, _, _ = O.refine_active(w, opts=O.options(**okw), max_outer=2)
    ran = []
    for mib in (1, 2, 4, 8, 16, 32, 64, 128, 1024):
        g, part = _dev(F, w)
        with F.Context(0, arena_bytes=mib << 20) as c:
            if call == "pair":
                st, _ = c.refine_pair(g, part, 4, 0, 1, w["eps"], w["alpha"], F.default_options(**okw), check=False)
            elif call == "batch":
                st, *_ = c.refine_batch(g, part, 4, w["eps"], w["alpha"], F.default_options(**okw), check=False)
            else:
                st, *_ = c.refine_active(g, part, 4, w["eps"], w["alpha"], F.default_options(**okw), max_outer=2,
                                         check=False)
        assert st in (0, F.FR_ERR_OOM)
        assert np.array_equal(part.cpu().numpy(), pref if st == 0 else np.array(w["part"], np.int32))
        ran.append(st == 0)
    assert ran == sorted(ran) and ran[-1]


def test_cluster_sizes_that_change(F):
    small, mid, big = I.grid2d_halves(32, 32, swaps=60), I.config(3, scale=1 / 64), I.config(4, scale=1 / 64)
    with F.Context(0) as c:
        for w in (small, mid, big, small, big, mid):
            for ctas in (0, 16, 4, 8):
                _batch(F, c, w, dict(cluster_ctas=ctas), mb=1)


@pytest.mark.parametrize("n,permille", [(700, 1000), (6000, 1000), (12000, 300)])
def test_fm_stacks_longer_than_their_ring(F, ctx, n, permille):
    w = I.rgg2d_bisection(n=n, mean_degree=9.0, seed=n)
    w = dict(w, alpha=1.0)
    _pair(F, ctx, w, mb=1, fm_permille=permille)


@pytest.mark.parametrize("seed", [1, 2])
def test_fm_on_long_rows(F, ctx, seed):
    w = hub_workload(90 + seed, n=1500, hubs=8, deg_lo=33, deg_hi=100, k=4)
    _batch(F, ctx, w, mb=1, fm_permille=200)
