"""GPU: Jaccard labels where the second pass keeps one, two and three words of the most
frequent items out of its counters: universes of a few words (some sets holding
nearly every item), set sizes on both sides of 128, one tile of centres and more."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("universe", [40, 64, 65, 128, 190, 193, 300, 520, 1500])
@pytest.mark.parametrize("groups,size", [(30, 25), (400, 60), (400, 140), (9_000, 20)])
def test_labels_are_the_exact_argmax(geek, universe, groups, size):
    rng = np.random.default_rng(universe + groups + size)
    p = np.arange(1, universe + 1) ** -0.3
    p /= p.sum()
    size = min(size, universe * 3 // 4)
    base = [np.unique(rng.choice(universe, size, p=p)) for _ in range(groups)]
    rows = [b for b in base for _ in range(2)]  # each pair becomes a seed, if no other equals it
    for _ in range(300):  # half a centre and as many items at random; nearly everything; a few items
        b = base[int(rng.integers(groups))]
        kind = rng.integers(3)
        if kind == 0:
            r = np.union1d(b[rng.random(b.size) < 0.5], rng.choice(universe, b.size // 2 + 1))
        elif kind == 1:
            r = np.setdiff1d(np.arange(min(universe, 500)), rng.choice(universe, 5))
        else:
            r = rng.choice(universe, 3)
        rows.append(np.unique(r))
    off = np.zeros(len(rows) + 1, np.int64)
    off[1:] = np.cumsum([r.size for r in rows])
    items = np.concatenate(rows).astype(np.uint32)
    ctx = geek.Context(0)
    u64 = lambda c: geek._dev(rng.integers(0, 1 << 63, c, dtype=np.uint64))  # noqa: E731
    data = ctx.sets(geek._dev(off), geek._dev(items.astype(np.int32)))
    bk = ctx.hash(data, 4, 4, mh_a=u64(16), mh_b=u64(16))
    seeds = ctx.silk(bk, 2, 4, 2, u64(8), u64(8), u64(2), u64(2))
    labels = torch.empty(off.size - 1, dtype=torch.int32, device="cuda")
    _, cen = ctx.assign_ex(data, bk, seeds, labels)
    assert seeds.k > 0
    if groups > 8192 and universe > 1000:
        assert seeds.k > 8192
    f = max(0, off.size - 1 - 340)  # the mixtures and the pairs before them
    ref, _, _ = oracle.assign_jaccard(off[f:] - off[f], items[off[f]:], cen["item_off"].cpu().numpy(),
                                      cen["items"].cpu().numpy().view(np.uint32))
    assert np.array_equal(labels.cpu().numpy()[f:], ref)
