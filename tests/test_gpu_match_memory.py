"""GPU: categorical labels without room for the mask tables come from the direct forms
(every pair of values; the Jaccard engine for DOPH-reduced sets): the same labels,
modes and statistics."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _hetero(geek, ctx, rng):
    n, d, n_cat, K, L, Kc = 3_000, 5, 7, 2, 6, 1
    home = rng.integers(0, 40, n)
    x = (rng.standard_normal((40, d)) * 9)[home] + rng.standard_normal((n, d)) * 0.1
    tok = (home[:, None] * (1 + np.arange(n_cat)) + (rng.random((n, n_cat)) < 0.2)) % 50 + 50 * np.arange(n_cat)
    data = ctx.hetero(geek._dev(x.astype(np.float32)), geek._dev(tok.astype(np.int32)))
    u64 = lambda c: geek._dev(rng.integers(0, 1 << 63, c, dtype=np.uint64))  # noqa: E731
    a = geek._dev(rng.standard_normal((K * L, d)).astype(np.float32))
    return data, ctx.hash(data, K, L, a=a, b=torch.zeros(K * L, device="cuda"), w=4.0, mh_a=u64(L * Kc), mh_b=u64(L * Kc), Kc=Kc)


def _doph(geek, ctx, rng):
    base = [np.unique(rng.integers(0, 5000, 40)) for _ in range(60)]
    rows = [np.unique(np.where(rng.random(b.size) < 0.9, b, rng.integers(0, 5000, b.size))) for b in base for _ in range(40)]
    off = np.zeros(len(rows) + 1, np.int64)
    off[1:] = np.cumsum([r.size for r in rows])
    data = ctx.sets(geek._dev(off), geek._dev(np.concatenate(rows).astype(np.int32)))
    u64 = lambda c: geek._dev(rng.integers(0, 1 << 63, c, dtype=np.uint64))  # noqa: E731
    return data, ctx.hash(data, 2, 8, mh_a=u64(16), mh_b=u64(16), doph_bins=48, doph_a=0x9E3779B97F4A7C15, doph_b=77)


@pytest.mark.parametrize("make", [_hetero, _doph])
def test_without_masks(geek, make):
    rng = np.random.default_rng(8)
    ctx = geek.Context(0)
    data, bk = make(geek, ctx, rng)
    u64 = lambda c: geek._dev(rng.integers(0, 1 << 63, c, dtype=np.uint64))  # noqa: E731
    seeds = ctx.silk(bk, 2, 6, 2, u64(12), u64(12), u64(2), u64(2))
    assert seeds.k > 1

    def assign():
        lab = torch.full((bk.n,), -7, dtype=torch.int32, device="cuda")
        st, cen = ctx.assign_ex(data, bk, seeds, lab)
        return lab, cen["modes"], st.sse

    want, went_on = assign(), 0
    for after in range(80):
        ctx.set_option(geek.OPT_TEST_FAIL_ALLOC, after)
        try:
            got = assign()
        except geek.GeekError as e:
            assert e.status == geek.ERR_NOMEM
            continue
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1]) and got[2] == want[2]
        try:  # raises while the countdown still runs
            for _ in range(80):
                assign()
            went_on += 1
        except geek.GeekError as e:
            assert e.status == geek.ERR_NOMEM
        ctx.set_option(geek.OPT_TEST_FAIL_ALLOC, -1)
    assert went_on >= 4  # each of the tables
