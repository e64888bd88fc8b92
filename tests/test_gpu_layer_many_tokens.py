"""Layer calls of more than 512 tokens in short segments: the base product of the CTA-pair kernel, so that a token without an
adapter has the bits of the base layer alone, and the oracle's values at a block's widths."""
import numpy as np
import pytest
import torch

import moin_inputs as mi
import paper_2410_09687_b200 as moin
from gpu_util import DEV, assert_layer_close, gpu_pool, oracle_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [513, 1030, 2048])
@pytest.mark.parametrize("shapes,r", [([(2048, 256)], 16), ([(704, 760)], 24), ([(2048, 2048), (2048, 256), (2048, 256)], 64),
                                      ([(2048, 5632), (2048, 5632)], 64), ([(5632, 2048)], 16)])
def test_segments(T, shapes, r):
    E = 7
    rng = mi.np_rng(T, r)
    te = np.repeat(rng.integers(-1, E, T // 6 + 1), 6)[:T].astype(np.int32)
    cases = [mi.layer_case(f"p{i}", T, d_in, d_out, mi.make_pool(E, r, d_in, d_out, 61, i, missing=(2,)), te, 2.0, 61, 5)
             for i, (d_in, d_out) in enumerate(shapes)]
    x = cases[0].x.to(DEV)
    Ws = [c.W.to(DEV) for c in cases]
    ys = [torch.empty(T, W.shape[0], dtype=torch.bfloat16, device=DEV) for W in Ws]
    plan = moin.plan_build(torch.from_numpy(te).to(DEV), E, moin.PLAN_SEGMENTS)
    moin.lora_linear_group(plan, moin.JobGroup([(x, W, gpu_pool(c.pool), y) for c, W, y in zip(cases, Ws, ys)]), 2.0)
    rows = np.unique(np.r_[0, T - 1, rng.integers(0, T, 40)])
    base = torch.from_numpy(np.nonzero((te == -1) | (te == 2))[0]).to(DEV)
    for c, W, y in zip(cases, Ws, ys):
        assert_layer_close(y[torch.from_numpy(rows).to(DEV)], oracle_layer(c, rows), c.name)
        assert torch.equal(y[base], moin.lora_linear(None, x, W, None, 0.0)[base])
    assert moin.device_status()["timeout_flag"] == 0
