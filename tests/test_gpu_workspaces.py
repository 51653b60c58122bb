"""What a call leaves in a context: the calls after it are admitted, and give the same results,
as without it."""
import numpy as np
import pytest

import oracle as O
from paper_1012_0006_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _dev(F, w):
    import torch
    return F.DeviceGraph.from_workload(w), torch.as_tensor(np.array(w["part"], np.int32)).cuda()


def _grid(nx, ny, k):
    w = dict(I.grid2d_halves(nx, ny, swaps=nx, alpha=2.0), mb=1)
    w["part"] = I.rcb(I.grid2d(nx, ny)[2], w["vwgt"], k)
    I.noise(w["xadj"], w["adjncy"], w["vwgt"], k, w["part"], 2 * nx, 7)
    w["k"] = k
    return w


@pytest.mark.parametrize("ctas", [4, 16])
def test_a_pair_call_leaves_room_for_a_sweep(gpu_lib, ctas):
    F = gpu_lib
    large, small = _grid(320, 300, 2), _grid(64, 61, 16)
    st, pref, _, _ = O.refine_batch(small, opts=O.options(mb=1))
    assert st == 0
    admitted = {}
    for sched in (1, 0):   # the pair's own launches, or the queue kernel
        for mib in range(8, 400, 4):
            with F.Context(0, arena_bytes=mib << 20) as c:
                g, part = _dev(F, large)
                st0, _ = c.refine_pair(g, part, 2, 0, 1, large["eps"], large["alpha"],
                                       F.default_options(mb=1, cluster_ctas=ctas, sweep_sched=sched), check=False)
                g, part = _dev(F, small)
                st, *_ = c.refine_batch(g, part, 16, small["eps"], small["alpha"],
                                        F.default_options(mb=1, cluster_ctas=ctas), check=False)
            assert np.array_equal(part.cpu().numpy(), pref if st == 0 else np.array(small["part"], np.int32))
            admitted.setdefault(mib, []).append((st0, st))
    assert len({s for v in admitted.values() for s in v}) > 1   # the bounds reach from refused to admitted
    for mib, (own, queue) in admitted.items():
        assert own == queue, mib
