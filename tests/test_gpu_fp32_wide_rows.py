"""GPU: the FP32 assignment around 160 < d <= 208, where two blocks share an SM
with a narrower ring: labels at the edges of its chunks, rows with and without
16-byte alignment, one block per SM and more; and what an odd d costs there."""
import time

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,pad", [(159, 0), (160, 0), (161, 0), (163, 2), (164, 4), (176, 0), (177, 3), (180, 1), (191, 1), (192, 0),
                                   (193, 0), (200, 0), (200, 5), (207, 0), (208, 0), (208, 8), (209, 0)])
@pytest.mark.parametrize("n,k", [(19_500, 67), (300, 130)])
def test_labels(geek, n, d, pad, k):
    rng = np.random.default_rng(d + k)
    c = rng.standard_normal((k, d)) * 2
    c[k // 2] = c[1]  # an exact tie
    x = (c[rng.integers(0, k, n)] + rng.standard_normal((n, d))).astype(np.float32)
    full = np.full((n, d + pad), np.nan, np.float32)
    full[:, :d] = x
    ctx = geek.Context(0)
    lab = torch.empty(n, dtype=torch.int32, device="cuda")
    ctx.assign_centers(ctx.dense(geek._dev(full)[:, :d]), geek._dev(c), lab, precision=geek.PREC_FP32)
    ref, _ = oracle.assign_dense(x, c)
    assert np.array_equal(lab.cpu().numpy(), ref)


def test_one_more_coordinate(geek):
    g = torch.Generator(device="cuda").manual_seed(1)
    ctx, n, k = geek.Context(0), 1_000_000, 50
    lab = torch.empty(n, dtype=torch.int32, device="cuda")

    def fastest(d):
        c = torch.rand(k, d, generator=g, device="cuda") * 20 - 10
        x = c[torch.randint(0, k, (n,), generator=g, device="cuda")] + torch.randn(n, d, generator=g, device="cuda")
        data, c, t = ctx.dense(x), c.double(), []
        for _ in range(8):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            ctx.assign_centers(data, c, lab, precision=geek.PREC_FP32, stats=False)
            torch.cuda.synchronize()
            t.append(time.perf_counter() - t0)
        return min(t[2:])

    # half of the blocks and loads that stall made it 1.8 times; the coordinate, its
    # padding and 4-byte copies are less than 1.3
    assert fastest(161) < 1.5 * fastest(160)
