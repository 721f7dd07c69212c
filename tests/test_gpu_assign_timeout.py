"""GPU: a dense assignment that sorts its flagged rows (100,000 and more) reports
a look-back wait that ran out itself, not the next call on the context.  The
failure is injected as in test_gpu_failures.py: a radix-sort tile that never
publishes its count, waits of 1 ms."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stats", [True, False])
@pytest.mark.parametrize("prec", ["PREC_BF16", "PREC_BF16X3"])
def test_sort_of_flagged_rows_reports_its_timeout(geek, prec, stats):
    rng = np.random.default_rng(11)
    n, d = 140_000, 16
    # two interleaved groups of centres far from the origin: no row has one near centre
    base = rng.standard_normal((2, d)) * 5 + 600.0
    c = geek._dev(base[np.arange(80) % 2] + rng.standard_normal((80, d)) * 0.5)
    x = geek._dev((base[rng.integers(0, 2, n)] + rng.standard_normal((n, d))).astype(np.float32))
    ctx, p = geek.Context(0), getattr(geek, prec)

    def assign(**kw):
        labels = torch.full((n,), -7, dtype=torch.int32, device="cuda")
        st = ctx.assign_centers(ctx.dense(x), c, labels, precision=p, **kw)
        return labels, st

    want, st = assign()
    assert st.n_recheck_rows >= 100_000
    ctx.set_option(geek.OPT_WAIT_LIMIT_NS, 1_000_000)
    ctx.set_option(geek.OPT_TEST_STALL_TILE, 2)
    with pytest.raises(geek.GeekError) as e:
        assign(stats=stats)
    assert e.value.status == geek.ERR_TIMEOUT
    ctx.set_option(geek.OPT_TEST_STALL_TILE, -1)
    got, _ = assign(stats=stats)  # no word left behind
    assert torch.equal(got, want)
