"""Short-segment shrink of a few tokens: eight warps split the reduction up to sixteen tokens, four beyond; reductions that leave
some warps without work, ranks that end inside a group of rows."""
import numpy as np
import pytest
import torch

import moin_inputs as mi
import paper_2410_09687_b200 as moin
from gpu_util import assert_layer_close, oracle_layer, run_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 15, 16, 17])
@pytest.mark.parametrize("d_in,r", [(64, 8), (448, 24), (2048, 64), (5632, 128)])
def test_layer(T, d_in, r):
    rng = mi.np_rng(T, d_in)
    pool = mi.make_pool(6, r, d_in, 72, 17, r, missing=(2,))
    case = mi.layer_case("few", T, d_in, 72, pool, rng.integers(-1, 6, T).astype(np.int32) if T > 1 else np.zeros(1, np.int32), 2.0, 17, T)
    y, _ = run_layer(case, moin.PLAN_SEGMENTS)
    assert_layer_close(y, oracle_layer(case), f"{T} tokens, {d_in} inputs, rank {r}")
