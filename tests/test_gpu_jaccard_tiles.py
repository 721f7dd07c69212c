"""GPU: the Jaccard assignment of sparse sets at the sizes where its tiles,
counters and passes change: k around a tile of centres, sets of 1 item up to
just above the counters' largest set, sets unlike every centre (they leave the
pruned pass for the full one), exact ties, and item ids above the lookup
table's range."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2106_10515_gb300 import geek
    return geek


def _sets(rng, groups, lo, hi, universe, extra_sizes, shift):
    """Pairs of equal sets (each pair becomes a seed), then the sets to label."""
    p = np.arange(1, universe + 1) ** -0.8
    p /= p.sum()
    base = [np.unique(rng.choice(universe, int(rng.integers(lo, hi)), p=p)) for _ in range(groups)]
    rows = [b for b in base for _ in range(2)]
    first = len(rows)
    for s in extra_sizes:
        b = base[int(rng.integers(groups))]
        kind = rng.integers(4)
        if kind == 0:  # near a centre
            r = b[rng.random(b.size) < 0.7]
        elif kind == 1:  # frequent items only: unlike every centre
            r = rng.choice(2 * s, s, replace=False)
        elif kind == 2:  # an equal mixture of two centres: ties
            c = base[int(rng.integers(groups))]
            r = np.union1d(b[: b.size // 2], c[: c.size // 2])
        else:  # items no centre holds
            r = universe + rng.choice(4 * s, s, replace=False)
        if kind != 3 and r.size < s:
            r = np.union1d(r, universe + rng.choice(4 * s, s - r.size, replace=False))
        rows.append(np.unique(r[:s] if r.size > s else r))
    off = np.zeros(len(rows) + 1, np.int64)
    off[1:] = np.cumsum([r.size for r in rows])
    items = (np.concatenate(rows) + shift).astype(np.uint32)
    return off, items, first


@pytest.mark.parametrize("groups,lo,hi,sizes,shift", [
    (3, 4, 20, (1, 2, 127, 128), 0),
    (513, 10, 60, (1, 5, 60, 128), 0),
    (513, 10, 60, (1, 5, 60, 128), 1 << 30),
    (257, 20, 300, (1, 129, 511, 512, 513), 0),
    (8250, 20, 70, (1, 30, 90, 128), 0),
])
def test_labels_are_the_exact_argmax(G, groups, lo, hi, sizes, shift):
    rng = np.random.default_rng(groups + hi)
    extra = [int(s) for s in rng.choice(sizes, 240)]
    off, items, first = _sets(rng, groups, lo, hi, 3000, extra, shift)
    n = off.size - 1
    ctx = G.Context(0)
    u64 = lambda c: G._dev(rng.integers(0, 1 << 63, c, dtype=np.uint64))  # noqa: E731
    data = ctx.sets(G._dev(off), G._dev(items.astype(np.int64).astype(np.int32)))
    bk = ctx.hash(data, 4, 4, mh_a=u64(16), mh_b=u64(16))
    seeds = ctx.silk(bk, 2, 4, 2, u64(8), u64(8), u64(2), u64(2))
    labels = torch.empty(n, dtype=torch.int32, device="cuda")
    _, cen = ctx.assign_ex(data, bk, seeds, labels)
    assert seeds.k > 0.97 * groups  # nearly every pair is a seed
    if groups > 8192:
        assert seeds.k > 8192       # more than one tile of centres
    coff = cen["item_off"].cpu().numpy()
    cit = cen["items"].cpu().numpy().view(np.uint32)
    # the extra sets and the pairs around them
    f = max(0, first - 40)
    ref, _, _ = oracle.assign_jaccard(off[f:] - off[f], items[off[f]:], coff, cit)
    assert np.array_equal(labels.cpu().numpy()[f:], ref)
