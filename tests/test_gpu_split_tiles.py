"""GPU: the split (three-product) assignment around its tiles: rows around a
tile of 128, centres around 128 and 256, each number of column blocks of the
stored halves, and row counts that leave units to the last blocks."""
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


@pytest.mark.parametrize("n,d,k", [(1, 16, 1), (127, 16, 127), (128, 33, 128), (129, 64, 129), (255, 65, 255),
                                   (257, 96, 256), (1000, 128, 257), (300, 127, 511), (500, 100, 513),
                                   (19_457, 128, 700), (40_000, 24, 1030)])
def test_labels_and_sse(G, n, d, k):
    rng = np.random.default_rng(n + d + k)
    x = rng.standard_normal((n, d)).astype(np.float32)
    c = rng.standard_normal((k, d))
    ctx = G.Context(0)
    lab_ref, dist = oracle.assign_dense(x, c)
    labels = torch.empty(n, dtype=torch.int32, device="cuda")
    st = ctx.assign_centers(ctx.dense(G._dev(x)), G._dev(c), labels, precision=G.PREC_BF16X3)
    assert np.array_equal(labels.cpu().numpy(), lab_ref)
    assert abs(st.sse - dist.sum()) <= 1e-6 * dist.sum()
