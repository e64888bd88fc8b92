"""Size queries against one another (host code, no GPU): a workspace sized for a batch serves every smaller one."""
import pytest


@pytest.mark.parametrize("query", ["moin_route_workspace_bytes", "moin_route_top2_workspace_bytes"])
@pytest.mark.parametrize("K,D", [(1, 8), (500, 768), (513, 64), (1000, 768), (5000, 768), (20000, 128), (6145, 8192), (700, 40)])
def test_router_scratch_grows_with_the_batch(query, K, D):
    import paper_2410_09687_b200 as moin
    from paper_2410_09687_b200 import build
    build.build()
    size = getattr(moin.lib(), query)
    sizes = [size(Q, K, D) for Q in list(range(0, 600)) + [1000, 1024, 4096, 65536]]
    assert all(a <= b for a, b in zip(sizes, sizes[1:]))
    assert sizes[-1] >= 65536 * 8
