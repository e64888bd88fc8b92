"""Handfuls of topics and narrow embeddings: both sides of the lines between the CUDA-core kernel, the cluster kernel and the
GEMM, with the runner-up."""
import numpy as np
import pytest
import torch

import moin_inputs as mi
import oracle
import paper_2410_09687_b200 as moin
from gpu_util import DEV, assert_router_matches

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Q,K,D", [
    (1, 1, 8), (7, 16, 768), (7, 17, 768), (40, 16, 776), (4095, 16, 64), (4096, 16, 64), (400, 2, 6144), (400, 2, 6152),   # few topics
    (384, 35, 40), (384, 36, 40), (385, 70, 40), (385, 71, 40), (1500, 140, 56), (1500, 141, 56), (2049, 300, 8)])          # narrow
def test_both_sides(Q, K, D):
    case = mi.planted_router(K=K, Q=Q, D=D, seed=80 + Q + K, unit_centroid_noise=True)
    router, q = moin.Router(case.centroids.to(DEV)), case.queries.to(DEV)
    ref = oracle.route(mi.bf16_bits(case.queries), mi.bf16_bits(case.centroids))
    cid, best = torch.empty(Q, dtype=torch.int32, device=DEV), torch.empty(Q, dtype=torch.float32, device=DEV)
    moin.route(router, q, out_centroid=cid, out_best_sim=best)
    assert_router_matches(cid.cpu().numpy(), ref)
    np.testing.assert_allclose(best.cpu().numpy(), ref["best"], atol=1e-5)   # fp32 sums of at most 6152 products
    static = torch.empty(Q, dtype=torch.int32, device=DEV)
    moin.route_static(router, q, static)
    assert torch.equal(static, cid)
    top = {k: v.cpu().numpy() for k, v in moin.route_top2(router, q).items()}
    assert_router_matches(top["centroid"], ref)
    if K == 1:
        assert (top["second"] == -1).all()
    else:
        assert (np.abs(top["margin"] - ref["margin"]) <= 2e-5).all() and (top["second"] != top["centroid"]).all()
    assert moin.device_status()["timeout_flag"] == 0
