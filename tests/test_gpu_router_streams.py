"""One centroid table, several calls in flight: a router serves the workers of a process, each on a stream of its own, and
graphs captured around a call replay beside them.  Every id has to be the one the call gives alone."""
import pytest
import torch

import moin_inputs as mi
import paper_2410_09687_b200 as moin
from gpu_util import DEV

pytestmark = pytest.mark.gpu

# single requests and small batches (the table in parts, in one part, the GEMM), and a batch that needs more scratch
SIZES = [(1, 5000, 768), (8, 5000, 768), (32, 1000, 256), (400, 500, 256), (512, 64, 64), (24, 500, 768)]


@pytest.mark.parametrize("explicit", [True, False])   # the stream as an argument, or the current one
def test_two_streams_one_router(explicit):
    for Q, K, D in SIZES:
        tables = mi.planted_router(K, 2 * Q * 8, D, Q + K, device=DEV)
        router = moin.Router(tables.centroids)
        batches = [tables.queries[i * Q:(i + 1) * Q].contiguous() for i in range(16)]
        alone = [moin.route(router, q) for q in batches]
        alone_margin = [moin.route_top2(router, q)["margin"] for q in batches]
        torch.cuda.synchronize()
        streams = [torch.cuda.Stream(), torch.cuda.Stream()]
        got, margins = [], []
        for rep in range(20):
            for i, q in enumerate(batches):
                s = streams[i % 2]
                out = torch.empty(Q, dtype=torch.int32, device=DEV)
                s.wait_stream(torch.cuda.current_stream())   # (the output's memory may have been the current stream's)
                if explicit:
                    moin.route(router, q, out_expert=out, stream=s)
                else:
                    with torch.cuda.stream(s):
                        moin.route(router, q, out_expert=out)
                        if rep % 4 == 0:
                            margins.append((i, moin.route_top2(router, q)["margin"]))
                got.append((i, out))
        torch.cuda.synchronize()
        assert all(torch.equal(out, alone[i]) for i, out in got), (Q, K, D)
        assert all(torch.equal(m, alone_margin[i]) for i, m in margins), (Q, K, D)
    assert moin.device_status()["timeout_flag"] == 0


def test_captured_single_request_after_larger_batches():
    case = mi.planted_router(5000, 4096, 768, 3, device=DEV)
    router = moin.Router(case.centroids)
    q = case.queries[:1].clone()
    out = torch.empty(1, dtype=torch.int32, device=DEV)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        moin.route(router, q, out_expert=out)
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        moin.route(router, q, out_expert=out)
    moin.route(router, case.queries)   # wants more scratch than the captured call had
    blocks = [torch.zeros(1 << 12, dtype=torch.uint8, device=DEV) for _ in range(64)]   # whoever gets freed scratch
    for i in range(1, 9):
        q.copy_(case.queries[i:i + 1])
        graph.replay()
        assert out.item() == case.labels[i].item()
    assert all(int(b.sum()) == 0 for b in blocks)
