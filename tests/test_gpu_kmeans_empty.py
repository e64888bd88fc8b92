"""K-means update where many clusters have no member: they keep their centroid, to the bit, and get its inverse norm,
wherever they lie among the others and however many there are."""
import numpy as np
import pytest
import torch

import moin_inputs as mi
import oracle
import paper_2410_09687_b200 as moin
from gpu_util import DEV

pytestmark = pytest.mark.gpu


def _assign(kind, N, K, rng):
    a = rng.integers(0, K, N)
    return {"one": np.full(N, K // 2), "none": np.full(N, -1), "front": a % max(1, K // 10), "back": K - 1 - a % max(1, K // 10),
            "every ninth": a // 9 * 9, "some points in none": np.where(a % 2 == 0, -1, a), "ends": a % 2 * (K - 1)}[kind].astype(np.int32)


@pytest.mark.parametrize("kind", ["one", "none", "front", "back", "every ninth", "some points in none", "ends"])
@pytest.mark.parametrize("N,K,D", [(700, 5000, 64), (3000, 1090, 768), (50, 33, 8), (900, 130, 1096), (1, 8, 256)])
def test_empty_clusters(kind, N, K, D):
    rng = np.random.default_rng(N + K)
    x = torch.from_numpy(rng.normal(size=(N, D)).astype(np.float32)).to(torch.bfloat16)
    c_old = torch.from_numpy(rng.normal(size=(K, D)).astype(np.float32)).to(torch.bfloat16)
    c_old[0] = 0   # an empty cluster with a zero row: inverse norm 0
    assign = _assign(kind, N, K, rng)
    plan = moin.plan_build(torch.from_numpy(assign).to(DEV), K, moin.PLAN_SEGMENTS)
    ref = oracle.kmeans_update(mi.bf16_bits(x), mi.bf16_bits(c_old), assign)["centroids"]
    old = c_old.to(DEV)
    inv = torch.full((K,), float("nan"), device=DEV)
    c_new = moin.kmeans_update(plan, x.to(DEV), old, inv_norm_new=inv)
    in_place = old.clone()
    moin.kmeans_update(plan, x.to(DEV), in_place, in_place)
    assert torch.equal(in_place, c_new)
    got = mi.bf16_to_f64(c_new.cpu())
    empty = np.ones(K, bool)
    empty[assign[assign >= 0]] = False
    assert np.array_equal(got[empty], mi.bf16_to_f64(c_old)[empty])
    # rounded once to bf16, from fp32 sums of at most 3000 values of size 1
    assert (np.abs(got - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-5).all()
    norms = np.sqrt((got ** 2).sum(1))
    want = np.divide(1.0, norms, out=np.zeros(K), where=norms > 0)
    np.testing.assert_allclose(inv.cpu().numpy(), want, rtol=2e-6)
