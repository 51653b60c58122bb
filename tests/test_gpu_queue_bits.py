"""The queue sweep's corridor bitmaps end with a group of 1,024 ids, whatever the number of
vertices: sweeps on device memory that held ones before, against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_1012_0006_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(9, 8), (33, 31), (32, 32), (41, 25), (64, 33)])
def test_sweep_on_used_memory(gpu_lib, nx, ny):
    import torch
    F = gpu_lib
    torch.cuda.empty_cache()
    used = torch.full((1 << 28,), -1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    del used
    torch.cuda.empty_cache()
    w = I.grid2d_halves(nx, ny, swaps=nx, alpha=4.0)
    w["part"] = I.rcb(I.grid2d(nx, ny)[2], w["vwgt"], 4)
    I.noise(w["xadj"], w["adjncy"], w["vwgt"], 4, w["part"], nx, 7)
    w["k"] = 4
    st, pref, rref, _ = O.refine_batch(w, opts=O.options(mb=1))
    assert st == 0
    g = F.DeviceGraph.from_workload(w)
    part = torch.as_tensor(np.array(w["part"], np.int32)).cuda()
    with F.Context(0) as ctx:
        st, res, _ = ctx.refine_batch(g, part, 4, w["eps"], w["alpha"], F.default_options(mb=1))
    assert [r["corridor_n"] for r in res] == [r["corridor_n"] for r in rref]
    assert np.array_equal(part.cpu().numpy(), pref)
