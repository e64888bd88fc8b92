"""Router GEMM: centroid norms that differ by powers of two from column to column and from tile to tile, several column
tiles one after the other in a CTA pair with little to multiply - a norm of another tile would change ids and cosines."""
import numpy as np
import pytest
import torch

import moin_inputs as mi
import oracle
import paper_2410_09687_b200 as moin
from gpu_util import DEV, assert_router_matches

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Q,K", [(4096, 5000), (2000, 4999)])
def test_norms_of_every_tile(Q, K):
    case = mi.planted_router(K=K, Q=Q, D=64, seed=90 + K)
    power = np.random.default_rng(K).integers(-3, 4, K) + (np.arange(K) // 64 % 2) * 8
    c = (case.centroids.float() * torch.from_numpy(2.0 ** power).float()[:, None]).to(torch.bfloat16)   # (exact)
    router, q = moin.Router(c.to(DEV)), case.queries.to(DEV)
    cid, best = torch.empty(Q, dtype=torch.int32, device=DEV), torch.empty(Q, dtype=torch.float32, device=DEV)
    moin.route(router, q, out_centroid=cid, out_best_sim=best)
    ref = oracle.route(mi.bf16_bits(case.queries), mi.bf16_bits(c))
    assert_router_matches(cid.cpu().numpy(), ref)
    # fp32 sums of 64 products and two reciprocal roots of 2^-22 relative error each
    np.testing.assert_allclose(best.cpu().numpy(), ref["best"], atol=1e-5)
    cid2, best2 = torch.empty_like(cid), torch.empty_like(best)
    for _ in range(20):
        moin.route(router, q, out_centroid=cid2, out_best_sim=best2)
        assert torch.equal(cid2, cid) and torch.equal(best2, best)
    top = moin.route_top2(router, q)
    assert torch.equal(top["centroid"], cid)
    assert (np.abs(top["margin"].cpu().numpy() - ref["margin"]) <= 2e-5).all()
    assert moin.device_status()["timeout_flag"] == 0
