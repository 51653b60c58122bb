"""Rounds with more pairs than clusters: a cluster scans the boundary candidates for its next
pair while the others commit theirs to the same list.  One cluster, two, and as many as fit,
against the oracle (whole numbers, equal)."""
import numpy as np
import pytest

import oracle as O
from paper_1012_0006_gb300 import inputs as I

pytestmark = pytest.mark.gpu

FIELDS = ("a", "b", "round", "accepted", "iters", "flow", "cut_before", "cut_after", "wA_after", "wB_after",
          "corridor_n", "corridor_arcs", "cut_fm", "fm_moves")


@pytest.mark.parametrize("ctas,clusters", [(4, 1), (4, 2), (16, 1), (16, 0), (0, 0)])
@pytest.mark.parametrize("fm", [0, 50])
def test_more_pairs_than_clusters(gpu_lib, ctas, clusters, fm):
    import torch
    F = gpu_lib
    w = I.rgg3d_rcb(n=24001, k=48, noise_ppm=40000, eps=0.03, alpha=2.0)
    _, _, pr, _ = O.rounds(w)
    assert np.bincount(np.asarray(pr)).max() > 12   # pairs of one round
    okw = dict(mb=1, adaptive=1, max_iters=4, alpha_max=8.0, fm_permille=fm)
    st, pref, rref, nref = O.refine_active(w, opts=O.options(**okw), max_outer=2)
    assert st == 0
    g = F.DeviceGraph.from_workload(w)
    part = torch.as_tensor(np.array(w["part"], np.int32)).cuda()
    with F.Context(0) as ctx:
        opts = F.default_options(cluster_ctas=ctas, grid_blocks=clusters * ctas, **okw)
        st, res, _, nouter = ctx.refine_active(g, part, w["k"], w["eps"], w["alpha"], opts, max_outer=2)
    assert nouter == nref and len(res) == len(rref)
    for rg, rc in zip(res, rref):
        for f in FIELDS:
            assert rg[f] == rc[f], (f, rg["a"], rg["b"], rg["round"])
    assert np.array_equal(part.cpu().numpy(), pref)


@pytest.mark.parametrize("offset", [0, 1, 3])
@pytest.mark.parametrize("n", [32767, 40001])
def test_a_round_that_is_taken_back(gpu_lib, n, offset):
    """Rounds of which a pair outgrows its cluster after others committed: the partition (at any
    multiple of four bytes) and the block weights are those before the round."""
    import torch
    F = gpu_lib
    w = I.rgg3d_rcb(n=n, k=6, noise_ppm=40000, eps=1.2, alpha=1.0)
    w["part"] = np.where(np.asarray(w["part"]) == 5, 4, w["part"]).astype(np.int32)   # uneven: large and small pairs
    okw = dict(mb=1)
    st, pref, rref, _ = O.refine_active(w, opts=O.options(**okw), max_outer=2)
    assert st == 0
    g = F.DeviceGraph.from_workload(w)
    store = torch.zeros(n + 8, dtype=torch.int32, device="cuda")
    part = store[offset:offset + n]
    part.copy_(torch.as_tensor(np.array(w["part"], np.int32)))
    with F.Context(0) as ctx:
        st, res, _, _ = ctx.refine_active(g, part, w["k"], w["eps"], w["alpha"],
                                          F.default_options(cluster_ctas=4, **okw), max_outer=2)
    assert len(res) == len(rref)
    for rg, rc in zip(res, rref):
        for f in FIELDS[:10]:
            assert rg[f] == rc[f], (f, rg["a"], rg["b"])
    assert np.array_equal(part.cpu().numpy(), pref)
