"""GPU: the BF16 assignment over pairs of row tiles (from 608 pairs of 256 rows on,
against 2,048 centres or more): row counts that end in a whole pair, in one tile
and inside a tile, on both sides of the rule; dimensions around a k-step."""
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


@pytest.mark.parametrize("d,k", [(8, 2047), (8, 2048), (17, 2304), (64, 2305), (70, 2100), (128, 2050)])
@pytest.mark.parametrize("n", [155_392, 155_393, 155_648, 155_649, 155_777, 156_031])
def test_labels(G, n, d, k):
    rng = np.random.default_rng(n + k)
    x = rng.standard_normal((n, d)).astype(np.float32)
    c = rng.standard_normal((k, d))
    ctx = G.Context(0)
    lab_ref, _ = oracle.assign_dense(x, c)
    labels = torch.empty(n, dtype=torch.int32, device="cuda")
    ctx.assign_centers(ctx.dense(G._dev(x)), G._dev(c), labels, precision=G.PREC_BF16)
    assert np.array_equal(labels.cpu().numpy(), lab_ref)
