"""GPU: the decision of flagged rows among their candidates, at the sizes where
its masks, tiles and waves change: centre counts around a word, a tile and a
list of 1,024, dimensions around a chunk of 32 and without 16-byte rows, few
and many flagged rows (both orders), centres too close for the FP32 distances,
and rows that are not finite."""
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


def _close_centres(rng, n, d, k, apart, off):
    """k centres in groups of up to 40 at distance ~apart, groups and points far
    from the origin (cancellation in |c|^2 - 2 x.c); points between the centres
    of a group."""
    groups = max(1, k // 40)
    base = rng.standard_normal((groups, d)) * 5 + off
    c = base[np.arange(k) % groups] + rng.standard_normal((k, d)) * apart
    x = base[rng.integers(0, groups, n)] + rng.standard_normal((n, d)) * 2 * apart
    return x.astype(np.float32), c


@pytest.mark.parametrize("prec", ["BF16", "BF16X3"])
@pytest.mark.parametrize("n,d,k", [(1, 8, 2), (127, 1, 3), (129, 7, 31), (1000, 31, 32), (1000, 33, 33), (700, 64, 255),
                                   (700, 65, 257), (500, 100, 1024), (300, 127, 1025), (600, 128, 1300),
                                   (140_000, 16, 80), (120_001, 30, 45)])
def test_flagged_rows_get_the_exact_label(G, prec, n, d, k):
    rng = np.random.default_rng(n + d + k)
    x, c = _close_centres(rng, n, d, k, 0.5, 60.0)
    ctx = G.Context(0)
    lab_ref, _ = oracle.assign_dense(x, c)
    labels = torch.empty(n, dtype=torch.int32, device="cuda")
    st = ctx.assign_centers(ctx.dense(G._dev(x)), G._dev(c), labels, precision=getattr(G, "PREC_" + prec))
    assert np.array_equal(labels.cpu().numpy(), lab_ref)
    if n > 1000 and prec == "BF16":
        assert st.n_recheck_rows > 100_000


@pytest.mark.parametrize("n", [3000, 130_000])
def test_left_over_rows(G, n):
    """Equal and nearly equal centres (no FP32 distance tells them apart), rows
    with infinities and NaN, and rows whose products overflow FP32."""
    rng = np.random.default_rng(n)
    d, k = 24, 120
    x, c = _close_centres(rng, n, d, k, 0.5, 60.0)
    c[60:90] = c[:30]
    c[90:] = c[:30] * (1 + 1e-9)
    x[5, 3], x[6, 0], x[7, 1] = np.inf, np.nan, -np.inf
    x[8] = 1e30
    ctx = G.Context(0)
    keep = np.ones(n, bool)
    keep[[5, 6, 7, 8]] = False
    lab_ref, _ = oracle.assign_dense(x, c)
    for prec in (G.PREC_BF16, G.PREC_BF16X3):
        labels = torch.empty(n, dtype=torch.int32, device="cuda")
        st = ctx.assign_centers(ctx.dense(G._dev(x)), G._dev(c), labels, precision=prec)
        got = labels.cpu().numpy()
        assert np.array_equal(got[keep], lab_ref[keep])
        assert (got[[5, 6, 7]] == -1).all()
        assert st.n_fp64_rows > 0
