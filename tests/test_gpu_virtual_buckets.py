"""GPU: SILK at bucket counts around the tile that one block lists (2,048), with
one-object buckets and buckets of two and more mixed in every proportion."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2106_10515_gb300 import geek
    return geek


@pytest.mark.parametrize("share", [0.0, 0.3, 1.0])
@pytest.mark.parametrize("n", [1, 2, 33, 1023, 1024, 1025, 2047, 2048, 2049, 6145])
def test_seeds(G, n, share):
    rng = np.random.default_rng(n)
    d, K, L, delta = 6, 2, 2, 2
    x = rng.uniform(-1e4, 1e4, (n, d))
    twins = np.flatnonzero(rng.random(n) < share)
    x[twins] = x[twins // 3 * 3]  # up to three rows alike
    x = x.astype(np.float32)
    a = rng.standard_normal((K * L, d)).astype(np.float32)
    b = rng.uniform(0, 1, K * L).astype(np.float32)
    sp = dict(Ks=2, Ls=4, delta=delta, mh_a=synth._u64(rng, 8), mh_b=synth._u64(rng, 8), dd_a=synth._u64(rng, 2),
              dd_b=synth._u64(rng, 2))
    ctx = G.Context(0)
    bk = ctx.hash(ctx.dense(G._dev(x)), K, L, a=G._dev(a), b=G._dev(b), w=1.0)
    seeds = ctx.silk(bk, **G.silk_args(sp))
    _, ref = oracle.hash_dense(x, a, b, 1.0, K, L)
    assert seeds.sets() == oracle.silk_on(ref, sp).sets()
