"""GPU: the centres' conversions at the counts where a warp takes one, four or more
centres (4,096; 9,728 per step) and around them: labels are the FP64 nearest centre
in every arithmetic, with the largest and the last centre among the winners, and many
centres cost no more than a few times their bytes."""
import time

import pytest
import torch

pytestmark = pytest.mark.gpu


def _nearest(x, c):
    """FP64 nearest centre of rows whose centre is known but for a few."""
    lab = torch.empty(x.shape[0], dtype=torch.int32, device="cuda")
    for s in range(0, x.shape[0], 16):
        lab[s:s + 16] = (x[s:s + 16, None].double() - c[None]).square_().sum(2).argmin(1).int()
    return lab


@pytest.mark.parametrize("prec", ["PREC_FP32", "PREC_BF16", "PREC_BF16X3"])
@pytest.mark.parametrize("k,d", [(1, 3), (31, 128), (4_095, 100), (4_096, 7), (4_097, 65), (19_455, 33), (19_457, 128), (78_001, 17),
                                 (200_003, 64)])
def test_labels(geek, prec, k, d):
    g = torch.Generator(device="cuda").manual_seed(k)
    c = torch.randn(k, d, generator=g, device="cuda", dtype=torch.float64) * 3
    c[k // 2] *= 1000  # the largest norm, by far
    at = torch.randint(0, k, (300,), generator=g, device="cuda")
    at[:4] = torch.tensor([0, k - 1, k // 2, k // 3], device="cuda")
    x = (c[at] + 0.3 * torch.randn(300, d, generator=g, device="cuda")).float()
    ctx = geek.Context(0)
    lab = torch.empty(300, dtype=torch.int32, device="cuda")
    ctx.assign_centers(ctx.dense(x), c, lab, precision=getattr(geek, prec))
    assert torch.equal(lab, _nearest(x, c))


def test_many_centres_few_rows(geek):
    g = torch.Generator(device="cuda").manual_seed(1)
    ctx = geek.Context(0)

    def fastest(k):
        c = torch.randn(k, 32, generator=g, device="cuda", dtype=torch.float64) * 50
        x, t = (c[:128] + 1).float(), []
        lab = torch.empty(128, dtype=torch.int32, device="cuda")
        for _ in range(6):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            ctx.assign_centers(ctx.dense(x), c, lab, precision=geek.PREC_BF16, stats=False)
            torch.cuda.synchronize()
            t.append(time.perf_counter() - t0)
        return min(t[1:])

    # one row tile walks the centres at 3.0 ns each; their conversions take 0.6 ns, and
    # 2.5 with a warp and its FP64 sum for each
    assert fastest(1_500_000) - fastest(500_000) < 1e6 * 4.6e-9
