"""Routing without scratch: the forms that moin_route takes for small problems when it is given no workspace, and
moin_route_static always - the same bits as with one, for the shapes that were ever served that way, and no shared state, so
that calls without a workspace may overlap."""
import ctypes

import numpy as np
import pytest
import torch

import moin_inputs as mi
import oracle
import paper_2410_09687_b200 as moin
from paper_2410_09687_b200 import binding
from gpu_util import DEV, assert_router_matches

pytestmark = pytest.mark.gpu

# cluster kernel (one part; parts of equal and of unequal numbers of tiles, with the reduction split or not; rows too long for
# 32 queries), GEMM (one column tile of each width; several; more than one block of 256 rows; K above 1024 and above what the
# cluster kernel takes; long rows), CUDA cores
SHAPES = [(24, 500, 768), (1, 5000, 768), (8, 5000, 216), (32, 1025, 40), (100, 1030, 384), (3, 13000, 64), (12, 600, 3200),
          (400, 60, 64), (400, 190, 72), (513, 256, 768), (777, 300, 128), (1024, 1024, 768), (1024, 1000, 3168), (385, 1, 64),
          (2000, 30, 200), (9, 7000, 64), (16000, 4, 64)]


def _call(router, q, ws):
    Q = q.shape[0]
    e, c = (torch.full((Q,), -7, dtype=torch.int32, device=DEV) for _ in range(2))
    b = torch.full((Q,), 7.0, dtype=torch.float32, device=DEV)
    st = moin.lib().moin_route(ctypes.byref(router.c), q.data_ptr(), Q, e.data_ptr(), c.data_ptr(), b.data_ptr(),
                               None if ws is None else ws.data_ptr(), 0 if ws is None else ws.numel(), binding._stream(None))
    assert st == 0, st
    return e, c, b


@pytest.mark.parametrize("Q,K,D", SHAPES)
def test_same_bits_without_scratch(Q, K, D):
    case = mi.planted_router(K=K, Q=Q, D=D, seed=60 + Q, unit_centroid_noise=True)
    cmap = torch.from_numpy(np.random.default_rng(Q).permutation(K).astype(np.int32)).to(DEV)
    centroids = case.centroids.clone()
    if K > 3:
        centroids[K // 2] = 0            # never chosen
        centroids[K - 1] = centroids[0]  # an exact tie: the lower index
    queries = case.queries.clone()
    if Q > 2:
        queries[Q // 2] = 0              # nothing wins
    router, q = moin.Router(centroids.to(DEV), cmap), queries.to(DEV)
    with_ws = _call(router, q, router.workspace(Q))
    without = _call(router, q, None)
    e, c = torch.empty(Q, dtype=torch.int32, device=DEV), torch.empty(Q, dtype=torch.int32, device=DEV)
    b = torch.empty(Q, dtype=torch.float32, device=DEV)
    moin.route_static(router, q, e, c, b)
    for name, want, a, s in zip(("expert", "centroid", "cosine"), with_ws, without, (e, c, b)):
        assert torch.equal(want.view(torch.int32), a.view(torch.int32)), name   # (the zero query's cosine is NaN)
        assert torch.equal(want.view(torch.int32), s.view(torch.int32)), name
    assert torch.equal(_call(router, q, None)[0], moin.route(router, q))
    rows = np.setdiff1d(np.arange(Q), [Q // 2])[:2048] if Q > 2 else np.arange(Q)
    ref = oracle.route(mi.bf16_bits(queries[torch.from_numpy(rows)]), mi.bf16_bits(centroids))
    assert_router_matches(c.cpu().numpy()[rows], ref)
    assert moin.device_status()["timeout_flag"] == 0


@pytest.mark.parametrize("Q,K,D", [(24, 500, 768), (1, 5000, 768), (8, 5000, 216), (32, 1025, 40), (100, 1030, 384), (3, 12000, 64)])
def test_runner_up_without_scratch(Q, K, D):
    # the cluster kernel (up to 2 x 12 parts of 512 topics for a few queries), whose two forms give the same bits
    case = mi.planted_router(K=K, Q=Q, D=D, seed=61 + Q, unit_centroid_noise=True)
    router, q = moin.Router(case.centroids.to(DEV)), case.queries.to(DEV)
    want = moin.route_top2(router, q)
    got = {k: torch.full_like(v, 7) for k, v in want.items()}
    st = moin.lib().moin_route_top2(ctypes.byref(router.c), q.data_ptr(), Q, *[got[k].data_ptr() for k in ("expert", "centroid", "second", "best", "margin")],
                                    None, 0, binding._stream(None))
    assert st == 0 and all(torch.equal(got[k], want[k]) for k in want)
    ref = oracle.route(mi.bf16_bits(case.queries), mi.bf16_bits(case.centroids))
    assert_router_matches(got["centroid"].cpu().numpy(), ref)
    assert (np.abs(got["margin"].cpu().numpy() - ref["margin"]) <= 2e-5).all()


def test_static_calls_overlap():
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for Q, K, D in [(1, 5000, 768), (20, 600, 128), (400, 500, 256), (777, 300, 128)]:
        case = mi.planted_router(K, 16 * Q, D, Q, device=DEV)
        router = moin.Router(case.centroids)
        batches = [case.queries[i * Q:(i + 1) * Q].contiguous() for i in range(16)]
        alone = [moin.route(router, x) for x in batches]
        outs = [[torch.empty(Q, dtype=torch.int32, device=DEV) for _ in batches] for _ in range(20)]
        torch.cuda.synchronize()
        for rep in outs:
            for i, (x, o) in enumerate(zip(batches, rep)):
                moin.route_static(router, x, o, stream=streams[i % 2])
        torch.cuda.synchronize()
        assert all(torch.equal(o, alone[i]) for rep in outs for i, o in enumerate(rep)), (Q, K, D)


@pytest.mark.parametrize("Q,K,D", [(1025, 1000, 64), (1000, 1025, 64), (1024, 1024, 3176), (66, 1000, 3200), (65536, 1, 64)])
def test_refused_without_scratch_as_before(Q, K, D):
    # past 1024 x 1024 and 65 535 products, or rows past 3168
    router = moin.Router(torch.ones(K, D, dtype=torch.bfloat16, device=DEV))
    q = torch.ones(Q, D, dtype=torch.bfloat16, device=DEV)
    out = torch.empty(Q, dtype=torch.int32, device=DEV)
    served = Q == 66   # (few queries: the cluster kernel, as before)
    st = moin.lib().moin_route(ctypes.byref(router.c), q.data_ptr(), Q, out.data_ptr(), None, None, None, 0, binding._stream(None))
    assert (st == 0) == served
