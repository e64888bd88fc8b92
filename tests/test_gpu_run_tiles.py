"""Row tiles of the long-run GEMM that several runs share: run boundaries off the 128-row grid, tiles of more runs than one
tile takes, a run across the two CTAs of a pair, rows without an adapter beside rows with one, two projections whose pools
lack different adapters.  The scratch starts as NaN, so that a row read where none was written shows."""
import numpy as np
import pytest
import torch

import moin_inputs as mi
import paper_2410_09687_b200 as moin
from gpu_util import DEV, assert_layer_close, gpu_pool, oracle_layer

pytestmark = pytest.mark.gpu
rng = np.random.default_rng(77)


@pytest.mark.parametrize("name,lengths,experts,r", [
    ("two runs in a tile", [100, 200], [0, 1], 64),
    ("run across the pair", [60, 300, 70], [2, 1, 0], 16),
    ("runs of one expert apart", [100, 20, 90, 30, 200], [1, 0, 1, 2, 1], 24),
    ("four and five runs", [32, 32, 32, 32, 25, 26, 26, 25, 26], [0, 1, 2, 3, 4, 0, 1, 2, 3], 64),
    ("single rows", [1] * 300, list(rng.integers(-1, 5, 300)), 8),
    ("no adapter between", [90, 77, 90, 127, 1, 128], [-1, 0, -1, 3, -1, 4], 72),
    ("more than one plan launch", list(rng.integers(1, 160, 40)), list(rng.integers(-1, 5, 40)), 128),
    ("a boundary on the grid", [128, 127, 1, 256, 384, 5], [0, 1, 2, 0, 1, 0], 40)])
def test_runs_share_row_tiles(name, lengths, experts, r):
    te = np.repeat(np.asarray(experts, np.int32), lengths)
    T, d_in, E, scale = len(te), 192, 5, 2.0
    plan = moin.plan_build(torch.from_numpy(te).to(DEV), E, moin.PLAN_TILES)
    cases, jobs = [], []
    for d_out, missing in ((264, (3,)), (72, (0,))):
        pool = mi.make_pool(E, r, d_in, d_out, 51, d_out, missing=missing)
        cases.append(mi.layer_case("runs", T, d_in, d_out, pool, te, scale, 51, r))
        x = cases[0].x if jobs else cases[-1].x
        cases[-1].x = x
        jobs.append((jobs[0][0] if jobs else x.to(DEV), cases[-1].W.to(DEV), gpu_pool(pool),
                     torch.full((T, d_out), float("nan"), dtype=torch.bfloat16, device=DEV)))
    group = moin.JobGroup(jobs)
    ws = torch.full((group.workspace_bytes,), 255, dtype=torch.uint8, device=DEV)
    moin.lora_linear_group(plan, group, scale, workspace=ws)
    torch.cuda.synchronize()
    for case, job in zip(cases, jobs):
        assert_layer_close(job[3], oracle_layer(case), name)
    assert moin.device_status()["timeout_flag"] == 0
