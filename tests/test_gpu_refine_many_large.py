"""GPU: which clusters' centre sums are cut into segments: on both sides of the line
for one cluster, among many of one size and beside a far larger one, on one stream and
with a second; the sums are the sequential FP64 ones either way, and many large
clusters cost what their chains do."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,sizes", [(1, [16_384]), (1, [16_385]), (1, [16_420]), (3, [16_400] * 40), (24, [17_000] * 40), (5, [500_000] + [30_000] * 12),
                                     (2, [900_000] + [20_000] * 10 + [17_000] * 3), (40, [70_000, 18_500, 18_000, 16_385, 5]),
                                     (1, [16_400] * 300 + [16_384] * 3 + [100] * 40), (35, [100_000] * 3 + [50_000] * 4 + [24_000] * 8)])
def test_sums_are_sequential(geek, d, sizes):
    rng = np.random.default_rng(d + len(sizes))
    lab = rng.permutation(np.repeat(np.arange(len(sizes)), sizes)).astype(np.int32)
    mean = rng.standard_normal((len(sizes), d)) * 3
    x = (mean[lab] + rng.standard_normal((lab.size, d))).astype(np.float32)
    ctx = geek.Context(0)
    c, labels, xd = geek._dev(mean), geek._dev(lab), geek._dev(x)
    ctx.refine(ctx.dense(xd), c, labels, 1, stats=False)
    got = c.cpu().numpy()
    for j, m in enumerate(sizes):
        want = np.cumsum(x[lab == j].astype(np.float64), axis=0)[-1] / m
        assert np.array_equal(got[j], want), j


def test_many_large_clusters(geek):
    g = torch.Generator(device="cuda").manual_seed(2)
    d, k = 128, 60
    ctx = geek.Context(0)

    def update_ms(size):
        lab = torch.randperm(size * k, generator=g, device="cuda") % k
        c = torch.rand(k, d, generator=g, device="cuda") * 20 - 10
        x = c[lab] + torch.randn(size * k, d, generator=g, device="cuda")
        data, ms = ctx.dense(x), []
        for _ in range(4):
            cc, ll = c.double(), lab.int()
            ctx.timing(True)
            ctx.timing_reset()
            ctx.refine(data, cc, ll, 1, stats=False)
            ms.append(ctx.timing_get("kernel.update_centres")[0])
            ctx.timing(False)
        return min(ms[1:])

    # twice the members; their segments took six times as long as the chains of half
    assert update_ms(20_000) < 3 * update_ms(10_000)
