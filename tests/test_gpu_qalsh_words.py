"""GPU: Alg. 1 buckets from (rounded value, id) words: object counts around the
one-block sort, values of every magnitude, many objects with one rounded value,
and equal values of both signs of zero at the cuts."""
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


@pytest.mark.parametrize("kind", ["plain", "magnitudes", "same_rounded", "zeros"])
@pytest.mark.parametrize("n,t", [(2, 2), (33, 5), (5119, 64), (5120, 5120), (5121, 700), (16_385, 9)])
def test_parts_equal_the_exact_split(G, kind, n, t):
    rng = np.random.default_rng(n + len(kind))
    d, m = 12, 4
    x = rng.standard_normal((n, d)).astype(np.float32)
    if kind == "magnitudes":
        x *= np.exp2(rng.integers(-40, 40, (n, 1))).astype(np.float32)
    elif kind == "same_rounded":  # a few FP32 values for all objects
        x = (1000 + 1e-4 * x).astype(np.float32)
    elif kind == "zeros":
        x[rng.random(n) < 0.7] = 0.0
        x[rng.random(n) < 0.3] *= -0.0
    a = rng.standard_normal((m, d)).astype(np.float32)
    ctx = G.Context(0)
    got = ctx.hash(ctx.dense(G._dev(x)), 1, m, a=G._dev(a), proj=G.PROJ_QALSH, t=t).copy_out()
    _, ref = oracle.transform_alg1(x, a, t)
    for key, r in (("obj_bucket", ref.obj_bucket), ("bucket_off", ref.boff), ("members", ref.bmem)):
        assert np.array_equal(got[key].cpu().numpy(), r), key
