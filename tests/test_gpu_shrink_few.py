"""Short-segment shrink of a few tokens: eight adapter rows an item up to sixteen tokens, sixteen beyond, in the same order of the
sums; reductions that leave some warps without work, ranks that end inside a group of rows."""
import numpy as np
import pytest
import torch

import moin_inputs as mi
import paper_2410_09687_b200 as moin
from gpu_util import DEV, assert_layer_close, oracle_layer, run_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 15, 16, 17])
@pytest.mark.parametrize("d_in,r", [(64, 8), (448, 24), (2048, 64), (5632, 128)])
def test_layer(T, d_in, r):
    rng = mi.np_rng(T, d_in)
    pool = mi.make_pool(6, r, d_in, 72, 17, r, missing=(2,))
    case = mi.layer_case("few", T, d_in, 72, pool, rng.integers(-1, 6, T).astype(np.int32) if T > 1 else np.zeros(1, np.int32), 2.0, 17, T)
    y, _ = run_layer(case, moin.PLAN_SEGMENTS)
    assert_layer_close(y, oracle_layer(case), f"{T} tokens, {d_in} inputs, rank {r}")


@pytest.mark.parametrize("d_in,r", [(128, 8), (2048, 40), (5632, 128)])
def test_sums_do_not_depend_on_the_batch(d_in, r):
    """The second half of the reduction takes the first half off again, so that h is nothing but what the order of the sums
    leaves: the same bits for sixteen tokens alone and in front of tokens without an adapter."""
    T, E, d_out = 16, 3, 64
    gen = torch.Generator().manual_seed(d_in)
    half = lambda rows: torch.randn(rows, d_in // 2, generator=gen).bfloat16()
    a, u = half(E * r), half(T)
    A, x = torch.cat([a, a], 1).view(E, r, d_in), torch.cat([u, -u], 1)
    B = torch.randn(E, d_out, r, generator=gen).bfloat16()
    pool = moin.Pool(A.to(DEV), B.to(DEV), torch.arange(E, dtype=torch.int32, device=DEV))
    W = torch.zeros(d_out, d_in, dtype=torch.bfloat16, device=DEV)
    te = torch.arange(T, dtype=torch.int32) % E

    def run(more):
        ids = torch.cat([te, torch.full((more,), -1, dtype=torch.int32)]).to(DEV)
        return moin.lora_linear(moin.plan_build(ids, E, moin.PLAN_SEGMENTS), torch.cat([x, half(2 * more).view(more, d_in)]).to(DEV), W, pool, 2.0)[:T]

    y = run(0)
    assert y.any()
    assert torch.equal(y, run(1)) and torch.equal(y, run(20))
