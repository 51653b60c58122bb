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
