"""GPU: SILK on buckets around and above the size from which a warp signs a
bucket (31, 32, 33, 100 and hundreds of members beside one-object buckets), for
every number of functions per table and both claim rules."""
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


@pytest.mark.parametrize("Ks,Ls,delta", [(1, 3, 1), (2, 5, 2), (3, 7, 2), (4, 3, 1), (3, 4, 10)])
@pytest.mark.parametrize("slow", [False, True])
def test_seeds_with_buckets_of_every_size(G, Ks, Ls, delta, slow):
    rng = np.random.default_rng(10 * Ks + Ls)
    sizes = [1] * 60 + [2, 3, 31, 31, 32, 32, 33, 33, 34, 100, 129, 400, 700]
    d, K, L = 8, 2, 4
    centre = rng.uniform(-1000, 1000, (len(sizes), d))
    x = np.concatenate([np.repeat(c[None], s, 0) for c, s in zip(centre, sizes)])
    x += (rng.random(x.shape) < 0.02) * rng.uniform(-300, 300, x.shape)  # some members move to buckets of their own
    x = x[rng.permutation(x.shape[0])].astype(np.float32)
    a = rng.standard_normal((K * L, d)).astype(np.float32)
    b = rng.uniform(0, 4, K * L).astype(np.float32)
    sp = dict(Ks=Ks, Ls=Ls, delta=delta, mh_a=synth._u64(rng, Ks * Ls), mh_b=synth._u64(rng, Ks * Ls),
              dd_a=synth._u64(rng, Ks), dd_b=synth._u64(rng, Ks))
    if slow:  # functions that repeat values on neighbouring ids: no claims
        sp = synth.silk_params_slow(sp, "all")
    ctx = G.Context(0)
    bk = ctx.hash(ctx.dense(G._dev(x)), K, L, a=G._dev(a), b=G._dev(b), w=4.0)
    seeds = ctx.silk(bk, **G.silk_args(sp))
    _, ref = oracle.hash_dense(x, a, b, 4.0, K, L)
    assert seeds.sets() == oracle.silk_on(ref, sp).sets()
