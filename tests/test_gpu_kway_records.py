"""The k-way searches' vertex records (connection weights per block) and their queue in
shared memory, where they can go wrong: vertices next to more blocks than a record holds,
rows of the largest degree, searches with more entries and more undone moves than shared
memory keeps.  Against the oracle; partitions and totals are integers: bit-exact."""
import numpy as np
import pytest

import oracle as O
from paper_1012_0006_gb300 import inputs as I
from tests.hub_graph import hub_workload

pytestmark = pytest.mark.gpu


def _rgg(n, deg, k, seed):
    xadj, adj, coords = I.rgg(2, n, I.rgg_radius(2, n, deg), seed)
    n = len(xadj) - 1
    w = dict(n=n, nnz=len(adj), xadj=xadj, adjncy=adj, adjwgt=I.edge_weights(xadj, adj, 1, 1 + seed % 4, seed),
             vwgt=I.uniform_i32(n, 0, 3, seed ^ 0x22), k=k, eps=0.25, alpha=1.0, mb=0)
    w["part"] = I.rcb(coords, w["vwgt"], k)
    I.noise(xadj, adj, w["vwgt"], k, w["part"], n // 10, seed ^ 0x33)
    return w


CASES = {
    "one block around": lambda: _rgg(300, 6.0, 2, 1),
    "about eight blocks around": lambda: _rgg(1200, 14.0, 130, 2),
    "more than eight blocks around": lambda: _rgg(700, 24.0, 128, 3),
    "unit weights, many ties": lambda: _rgg(900, 16.0, 64, 4),
    "hubs of degree up to 900": lambda: hub_workload(5, n=1500, hubs=6, deg_lo=33, deg_hi=900, k=40, weighted=False),
    "hubs in few blocks": lambda: hub_workload(6, n=1500, hubs=6, deg_lo=31, deg_hi=66, k=3, weighted=False),
    "many entries": lambda: I.rgg3d_rcb(n=20011, k=9, noise_ppm=60000, seed=7, eps=0.1),
}


@pytest.mark.parametrize("alpha", [0, 10, 10**6])
@pytest.mark.parametrize("case", CASES)
def test_records(gpu_lib, case, alpha):
    import torch
    F = gpu_lib
    w = CASES[case]()
    g = F.DeviceGraph.from_workload(w)
    dev = lambda: torch.as_tensor(np.array(w["part"], np.int32)).cuda()  # noqa: E731
    pa, pb, pr, _ = O.rounds(w)
    pairs = [(int(a), int(b)) for a, b, r in zip(pa, pb, pr) if r == 0]
    with F.Context(0) as ctx:
        st, pref, tref, cref = O.multitry(w, pairs, alpha, seed=3)
        part = dev()
        st2, tot, changed = ctx.multitry(g, part, w["k"], w["eps"], pairs, alpha, seed=3)
        assert (st, st2) == (0, 0)
        assert {f: tot[f] for f in tref} == tref
        assert np.array_equal(part.cpu().numpy(), pref) and np.array_equal(changed, cref)
        for init in (0, 1):
            st, pref, tref, rref = O.kway_global(w, alpha=alpha, init_mode=init, max_rounds=3, seed=5)
            part = dev()
            st2, tot = ctx.kway_global(g, part, w["k"], w["eps"], init_mode=init, alpha=alpha, max_rounds=3, seed=5)
            assert (st, st2) == (0, 0)
            assert (tot["gain"], tot["tried"], tot["kept"], tot["searches"]) == \
                (tref["gain"], tref["tried"], tref["kept"], rref)
            assert np.array_equal(part.cpu().numpy(), pref)
