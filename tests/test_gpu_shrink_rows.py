"""Long-run shrink: rows dealt to lanes and warps for ranks that do not divide a warp, with the reduction in one part and cut
over clusters of two, four and eight; every run ends inside a row tile."""
import numpy as np
import pytest
import torch

import moin_inputs as mi
import paper_2410_09687_b200 as moin
from gpu_util import DEV, assert_layer_close, gpu_pool, oracle_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_proj,r", [(1, 8), (1, 120), (3, 24), (3, 80), (2, 128)])
@pytest.mark.parametrize("T", [150, 1700, 5000, 12000])   # reduction of 2048 cut in eight, four, two, one
def test_rows(T, n_proj, r):
    E, d_in, d_out = 5, 2048, 64
    lengths = [T // 2 - 3, T // 3 + 1]
    lengths.append(T - sum(lengths))
    te = np.repeat(np.array([3, 0, 1], np.int32), lengths)
    plan = moin.plan_build(torch.from_numpy(te).to(DEV), E, moin.PLAN_TILES)
    rng = mi.np_rng(T, r)
    ends = np.cumsum(lengths)
    rows = np.unique(np.r_[0, ends - 1, ends[:-1], rng.integers(0, T, 60)])
    cases = [mi.layer_case(f"p{i}", T, d_in, d_out, mi.make_pool(E, r, d_in, d_out, 41, i, missing=(i,) if n_proj > 1 else ()), te, 2.0, 41, 9)
             for i in range(n_proj)]
    x = cases[0].x.to(DEV)
    jobs = [(x, c.W.to(DEV), gpu_pool(c.pool), torch.empty(T, d_out, dtype=torch.bfloat16, device=DEV)) for c in cases]
    moin.lora_linear_group(plan, moin.JobGroup(jobs), 2.0)
    torch.cuda.synchronize()
    assert moin.device_status()["timeout_flag"] == 0
    for c, job in zip(cases, jobs):
        assert torch.equal(c.x, cases[0].x)
        assert_layer_close(job[3][torch.from_numpy(rows).to(DEV)], oracle_layer(c, rows), c.name)
