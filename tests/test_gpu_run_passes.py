"""Low-rank passes of the long-run GEMM over many tiles of one CTA pair: the table of a tile's passes is rewritten while
the tile before it is still multiplied, whatever the tile's last runs are."""
import numpy as np
import pytest
import torch

import moin_inputs as mi
import paper_2410_09687_b200 as moin
from gpu_util import DEV, assert_layer_close, gpu_pool, oracle_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("runs,experts", [
    ([90, 166], [0, -1]),                   # a tile's last pass has no adapter and so loads nothing
    ([40, 40, 48, 128], [-1, 2, -1, -1]),   # ... the second CTA's rows have none at all
    ([256, 200, 56], [-1, 1, 3]),           # no pass in every other tile (3: an expert without a slot)
])
def test_passes_without_adapter_over_many_tiles(runs, experts):
    # 64 columns to multiply and 8192 to make: a short main loop and about five tiles for each of the 74 CTA pairs
    d_in, d_out, r, E, n = 64, 8192, 8, 4, 2560
    reps = -(-n // sum(runs))
    te = np.repeat(np.asarray(experts * reps, np.int32), runs * reps)
    pool = mi.make_pool(E, r, d_in, d_out, 91, len(runs), std_a=0.2, std_b=0.2, missing=(3,))
    case = mi.layer_case("passes", len(te), d_in, d_out, pool, te, 2.0, 91)
    plan = moin.plan_build(torch.from_numpy(te).to(DEV), E, moin.PLAN_TILES)
    x, W, p = case.x.to(DEV), case.W.to(DEV), gpu_pool(pool)
    y = moin.lora_linear(plan, x, W, p, 2.0)
    assert_layer_close(y, oracle_layer(case))
    for _ in range(20):
        assert torch.equal(moin.lora_linear(plan, x, W, p, 2.0), y)
    assert moin.device_status()["timeout_flag"] == 0
