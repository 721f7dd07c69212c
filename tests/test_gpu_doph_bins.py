"""GPU: densification at bin counts around a mask word and sets from none to
more items than bins."""
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


@pytest.mark.parametrize("Dp", [1, 2, 31, 32, 33, 63, 65, 400, 1023, 1024])
def test_minhash_of_reduced_sets(G, Dp):
    rng = np.random.default_rng(Dp)
    sizes = np.concatenate([[0, 1, 1, 2, 0, 31, 32, 33, 2000], rng.integers(0, 80, 200)])
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    items = np.concatenate([np.sort(rng.choice(1 << 20, s, replace=False)) for s in sizes]).astype(np.uint32)
    K, L = 2, 3
    mh_a, mh_b = synth._u64(rng, K * L), synth._u64(rng, K * L)
    Ap, Bp = int(rng.integers(1, 1 << 62)) * 2 + 1, int(rng.integers(0, 1 << 62))
    ctx = G.Context(0)
    got = ctx.hash(ctx.sets(G._dev(off), G._dev(items.astype(np.int32))), K, L, mh_a=G._dev(mh_a), mh_b=G._dev(mh_b),
                   doph_bins=Dp, doph_a=Ap, doph_b=Bp).copy_out()
    _, mh, ref = oracle.transform_sparse_doph(off, items, Dp, Ap, Bp, mh_a, mh_b, K, L)
    assert np.array_equal(got["codes"].cpu().numpy().view(np.uint32), mh)
    assert np.array_equal(got["members"].cpu().numpy(), ref.bmem)
