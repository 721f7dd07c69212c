"""GPU: segments around the size that one block sorts (5,120) and scans around
16,384 values: tables of SRP codes in one and in two key words."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2106_10515_gb300 import geek
    return geek


@pytest.mark.parametrize("K", [1, 7, 64, 65, 100])
@pytest.mark.parametrize("n", [2, 31, 321, 5119, 5120, 5121, 16_384, 16_385])
def test_buckets(G, n, K):
    rng = np.random.default_rng(n + K)
    d, L = 6, 3
    x = rng.standard_normal((max(n // 3, 1), d))[rng.integers(0, max(n // 3, 1), n)].astype(np.float32)
    a = rng.standard_normal((K * L, d)).astype(np.float32)
    b = np.zeros(K * L, np.float32)
    ctx = G.Context(0)
    got = ctx.hash(ctx.dense(G._dev(x)), K, L, a=G._dev(a), b=G._dev(b), w=1.0, proj=G.PROJ_SRP).copy_out()
    _, ref = oracle.hash_dense(x, a, b, 1.0, K, L, proj="srp")
    for key, r in (("obj_bucket", ref.obj_bucket), ("bucket_off", ref.boff), ("members", ref.bmem)):
        assert np.array_equal(got[key].cpu().numpy(), r), key
