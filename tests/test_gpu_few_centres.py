"""GPU: tensor-core assignment to few centres, whose tiles are 64 and 128 wide: labels
around those counts, decided rows and candidates alike, and what few centres cost."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["PREC_BF16", "PREC_BF16X3"])
@pytest.mark.parametrize("k", [1, 2, 31, 63, 64, 65, 127, 128, 129, 256])
@pytest.mark.parametrize("n,d,off", [(700, 33, 0.0), (20_011, 100, 0.0), (3_001, 128, 30.0), (120_000, 64, 40.0)])
def test_labels(geek, prec, k, n, d, off):
    g = torch.Generator(device="cuda").manual_seed(k + d)
    c = torch.randn(k, d, generator=g, device="cuda") + off  # off: the window holds several centres
    x = c[torch.randint(0, k, (n,), generator=g, device="cuda")] + torch.randn(n, d, generator=g, device="cuda")
    ctx = geek.Context(0)
    want, got = (torch.full((n,), -7, dtype=torch.int32, device="cuda") for _ in range(2))
    ctx.assign_centers(ctx.dense(x), c.double(), want, precision=geek.PREC_FP32)
    ctx.assign_centers(ctx.dense(x), c.double(), got, precision=getattr(geek, prec))
    assert torch.equal(got, want)


def test_few_centres_cost_less(geek):
    g = torch.Generator(device="cuda").manual_seed(3)
    n, d = 2_000_000, 128
    ctx = geek.Context(0)
    lab = torch.empty(n, dtype=torch.int32, device="cuda")

    def pass_ms(k):
        c = torch.rand(k, d, generator=g, device="cuda") * 20 - 10
        x = c[torch.randint(0, k, (n,), generator=g, device="cuda")] + torch.randn(n, d, generator=g, device="cuda")
        data, ms = ctx.dense(x), []
        ctx.timing(True)
        for _ in range(6):
            ctx.timing_reset()
            ctx.assign_centers(data, c.double(), lab, precision=geek.PREC_BF16X3, stats=False)
            ms.append(ctx.timing_get("kernel.assign_tc")[0])
        ctx.timing(False)
        return min(ms[1:])

    # a tile of 64 columns against one of 256: 0.58; the same where both are 256 wide
    assert pass_ms(30) < 0.8 * pass_ms(250)
