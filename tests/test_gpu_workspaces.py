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


def _calls(F, c, w, sched, check=False):
    """Pairs and active scheduling with FM and multi-try, sweeps and k-way rounds in turn on one context;
    after each: its status, what the context holds, the partition."""
    k, out = w["k"], []
    for call in ("pair", "active", "batch", "fm", "kway", "pair", "batch", "active"):
        g, part = _dev(F, w)
        fm = dict(mb=1, fm_permille=50)
        if call == "pair":
            st, *_ = c.refine_pair(g, part, k, 0, 1, w["eps"], w["alpha"], F.default_options(**fm, sweep_sched=sched),
                                   check=check)
        elif call == "active":
            st, *_ = c.refine_active(g, part, k, w["eps"], w["alpha"],
                                     F.default_options(**fm, mt_alpha=10, sweep_sched=sched), max_outer=1, check=check)
        elif call == "batch":
            st, *_ = c.refine_batch(g, part, k, w["eps"], w["alpha"], F.default_options(mb=1, mb_reps=2), check=check)
        elif call == "fm":
            st, *_ = c.refine_batch(g, part, k, w["eps"], w["alpha"], F.default_options(**fm), check=check)
        else:
            st, _ = c.kway_global(g, part, k, w["eps"], init_mode=0, alpha=10, max_rounds=1, seed=1, check=check)
        out.append((st, c.workspace_bytes, part.cpu().numpy()))
    return out


def test_a_bounded_context_stays_within_its_bound(gpu_lib):
    F = gpu_lib
    w = _grid(160, 150, 8)
    with F.Context(0) as c:
        want = _calls(F, c, w, 1, check=True)
    start = np.array(w["part"], np.int32)
    seen = set()
    for mib in range(4, 420, 8):
        bound = mib << 20
        with F.Context(0, arena_bytes=bound) as c:
            own = _calls(F, c, w, 1)
        with F.Context(0, arena_bytes=bound) as c:
            queue = _calls(F, c, w, 0)
        for i in range(len(want)):
            assert queue[i][0] == own[i][0], (mib, i)   # admitted as with the round's own launches
            # (what those hold: the sweep arrays of an FM call are not added to its bound)
            assert queue[i][1] <= max(bound, own[i][1]), (mib, i)
            assert np.array_equal(queue[i][2], want[i][2] if queue[i][0] == 0 else start), (mib, i)
            seen.add(queue[i][0])
    assert seen == {0, F.FR_ERR_OOM}


def test_workspace_bytes_counts_what_is_held(gpu_lib):
    import torch
    F = gpu_lib
    w = _grid(700, 600, 8)
    with F.Context(0) as c:   # (kernels and contexts loaded before the count)
        _calls(F, c, w, 0, check=True)
    _, part = _dev(F, w)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    with F.Context(0) as c:
        _calls(F, c, w, 0, check=True)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        used, held = before - torch.cuda.mem_get_info()[0], c.workspace_bytes
    assert abs(used - held) < 32 << 20   # (device memory comes in blocks of 2 MiB)


def test_a_sweep_of_other_sizes_is_admitted_alone(gpu_lib):
    """A graph with many vertices and few pairs, then one with few vertices and many pairs: under
    a bound that holds the workspace of each, not one of both sizes together."""
    F = gpu_lib
    large, small = _grid(320, 300, 2), _grid(64, 61, 16)
    opts = F.default_options(mb=1, cluster_ctas=4)
    st, pref, _, _ = O.refine_batch(small, opts=O.options(mb=1))
    assert st == 0

    def sweep(c, w):
        g, part = _dev(F, w)
        st, *_ = c.refine_batch(g, part, w["k"], w["eps"], w["alpha"], opts, check=False)
        return st, part.cpu().numpy()

    seen = set()
    for mib in range(40, 240, 4):
        with F.Context(0, arena_bytes=mib << 20) as c:   # the large graph's arrays, no queue workspace of its
            g, part = _dev(F, large)
            c.refine_batch(g, part, 2, large["eps"], large["alpha"], F.default_options(mb=1, sweep_sched=1))
            alone = sweep(c, small)
        with F.Context(0, arena_bytes=mib << 20) as c:
            assert sweep(c, large)[0] == 0
            after = sweep(c, small)
            assert c.workspace_bytes <= mib << 20
        assert after[0] == alone[0], mib
        assert np.array_equal(after[1], pref if after[0] == 0 else np.array(small["part"], np.int32))
        seen.add(after[0])
    assert seen == {0, F.FR_ERR_OOM}
