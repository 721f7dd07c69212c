"""GPU: the assignment by most equal attributes (heterogeneous rows, DOPH
tokens) at the sizes where its bit masks and planes change: k around 32
centres per word, around one and two rounds of 32 words, attribute counts
around the planes' limits, rows that match no centre and exact ties."""
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


@pytest.fixture(scope="module")
def ctx(G):
    return G.Context(0)


@pytest.mark.parametrize("groups,n_cat,L", [(1, 1, 1), (31, 10, 8), (32, 3, 2), (33, 15, 8), (130, 23, 8),
                                            (1023, 9, 4), (1025, 24, 8), (2100, 5, 8)])
def test_hetero_labels(G, ctx, groups, n_cat, L):
    """Pairs of equal rows (each pair a seed), then rows that mix the
    attributes of several pairs, and rows with values nobody else has."""
    rng = np.random.default_rng(groups)
    K, Kc, d, extra = 2, 1, 4, 700
    gx = rng.uniform(-50, 50, (groups, d)).astype(np.float32)
    gt = rng.integers(0, 12, (groups, n_cat))
    x = np.concatenate([np.repeat(gx, 2, 0), gx[rng.integers(0, groups, extra)]])
    t = np.concatenate([np.repeat(gt, 2, 0),
                        np.stack([gt[rng.integers(0, groups, extra), j] for j in range(n_cat)], 1)])
    x[-60:] = 1000 + rng.uniform(0, 1e4, (60, d))
    t[-60:] = 12 + rng.integers(0, 5, (60, n_cat))
    tok = (t + 20 * np.arange(n_cat)).astype(np.int32)
    u64 = lambda c: G._dev(rng.integers(0, 1 << 63, c, dtype=np.uint64))  # noqa: E731
    data = ctx.hetero(G._dev(x), G._dev(tok))
    a = rng.standard_normal((K * L, d)).astype(np.float32)
    bk = ctx.hash(data, K, L, a=G._dev(a), b=G._dev(np.zeros(K * L, np.float32)), w=1.0, mh_a=u64(L * Kc),
                  mh_b=u64(L * Kc), Kc=Kc)
    seeds = ctx.silk(bk, 2, 6, 2, u64(12), u64(12), u64(2), u64(2))
    labels = torch.empty(x.shape[0], dtype=torch.int32, device="cuda")
    st, cen = ctx.assign_ex(data, bk, seeds, labels)
    if seeds.k == 0:  # one bucket in one table: no bin of two buckets, no seed
        assert groups == 1 and bool((labels == -1).all())
        return
    assert seeds.k >= 0.9 * groups
    codes = bk.copy_out()["codes"].cpu().numpy()
    ranks = [np.unique(codes[:, l * K:(l + 1) * K], axis=0, return_inverse=True)[1].reshape(-1) for l in range(L)]
    attrs = np.concatenate([np.stack(ranks, 1), tok], 1).astype(np.int64)
    modes = cen["modes"].cpu().numpy()
    m = np.zeros((attrs.shape[0], modes.shape[0]), np.int16)
    for j in range(attrs.shape[1]):
        m += attrs[:, j, None] == modes[None, :, j]
    assert np.array_equal(labels.cpu().numpy(), m.argmax(1))
    best = m.max(1).astype(np.float64)
    dist = 1 - best / (2 * attrs.shape[1] - best)
    assert abs(st.sse - dist.sum()) <= 1e-12 * dist.sum() and st.radius_max == dist.max()


@pytest.mark.parametrize("groups,D", [(5, 16), (40, 31), (40, 32), (70, 511), (70, 512), (33, 1024)])
def test_doph_labels(G, ctx, groups, D):
    rng = np.random.default_rng(D)
    base = [np.unique(rng.integers(0, 5000, int(rng.integers(3, 60)))) for _ in range(groups)]
    rows = [b for b in base for _ in range(2)]
    for _ in range(500):
        b = base[int(rng.integers(groups))]
        rows.append(np.union1d(b[rng.random(b.size) < 0.6], rng.integers(0, 5000, int(rng.integers(1, 20)))))
    off = np.zeros(len(rows) + 1, np.int64)
    off[1:] = np.cumsum([r.size for r in rows])
    items = np.concatenate(rows).astype(np.uint32)
    u64 = lambda c: G._dev(rng.integers(0, 1 << 63, c, dtype=np.uint64))  # noqa: E731
    Ap, Bp = int(rng.integers(1, 1 << 61)) * 2 + 1, int(rng.integers(0, 1 << 62))
    data = ctx.sets(G._dev(off), G._dev(items.astype(np.int32)))
    bk = ctx.hash(data, 3, 4, mh_a=u64(12), mh_b=u64(12), doph_bins=D, doph_a=Ap, doph_b=Bp)
    seeds = ctx.silk(bk, 2, 6, 2, u64(12), u64(12), u64(2), u64(2))
    labels = torch.empty(len(rows), dtype=torch.int32, device="cuda")
    _, cen = ctx.assign_ex(data, bk, seeds, labels)
    assert seeds.k >= 0.9 * groups
    tok = oracle.doph(off, items, D, Ap, Bp).reshape(len(rows), D).astype(np.uint64)
    modes = cen["modes"].cpu().numpy().view(np.uint64)
    m = (tok[:, None, :] == modes[None, :, :]).sum(2)
    assert np.array_equal(labels.cpu().numpy(), m.argmax(1))
