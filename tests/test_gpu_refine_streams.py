"""GPU: extra passes around the row count from which the small clusters' update
and the rows' conversion run on a second stream: centres and labels equal the
oracle's, also when the caller's next work reads them at once and when calls
follow each other on one stream without a wait."""
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


@pytest.mark.parametrize("prec", ["FP32", "BF16", "BF16X3"])
@pytest.mark.parametrize("n", [(1 << 20) - 1, 1 << 20, (1 << 20) + 129])
def test_centres_and_labels(G, n, prec):
    rng = np.random.default_rng(n)
    d, k, passes = 9, 150, 2
    p = np.full(k, 0.6 / (k - 2))
    p[0], p[1] = 0.37, 0.03  # one large cluster, one around the limit of a segment's
    c = rng.standard_normal((k, d)) * 4
    x = (c[rng.choice(k, n, p=p)] + rng.standard_normal((n, d))).astype(np.float32)
    c0 = c + rng.standard_normal((k, d)) * 0.3
    lab0, _ = oracle.assign_dense(x, c0)
    ctx = G.Context(0)
    with torch.cuda.stream(torch.cuda.Stream()):
        xd, got = G._dev(x), []
        for _ in range(3):
            cd, labels = G._dev(c0), G._dev(lab0.astype(np.int32))
            ctx.refine(ctx.dense(xd), cd, labels, passes, precision=getattr(G, "PREC_" + prec), stats=False)
            got.append((cd.clone(), labels.clone()))
    torch.cuda.synchronize()
    lab_ref, c_ref, _ = oracle.refine_passes(x, c0, lab0, passes)
    for cd, labels in got:
        assert np.array_equal(cd.cpu().numpy(), c_ref)
        assert np.array_equal(labels.cpu().numpy(), lab_ref)
