"""GPU: which row counts the BF16 assignment takes in pairs of row tiles: those whose
pairs come out about as even on the SMs as single tiles do; labels on both sides, with
a last pair of one row, of one tile and a row, and short of a row."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _assign(geek, ctx, x, c, prec):
    lab = torch.full((x.shape[0],), -7, dtype=torch.int32, device="cuda")
    ctx.assign_centers(ctx.dense(x), c, lab, precision=prec, stats=False)
    return lab


@pytest.mark.parametrize("n", [310_401, 311_041, 311_169, 311_295, 311_297])
@pytest.mark.parametrize("d,k", [(64, 2_048), (70, 2_049), (128, 2_300)])
def test_labels(geek, n, d, k):
    g = torch.Generator(device="cuda").manual_seed(n + d)
    x = torch.randn(n, d, generator=g, device="cuda")
    c = torch.randn(k, d, generator=g, device="cuda", dtype=torch.float64)
    ctx = geek.Context(0)
    assert torch.equal(_assign(geek, ctx, x, c, geek.PREC_BF16), _assign(geek, ctx, x, c, geek.PREC_FP32))


# (n, d, k, pairs): 152 SMs take 16 rounds of single tiles where 8 of pairs do, 17 where 9 of pairs, ...
@pytest.mark.parametrize("n,d,k,pairs", [(156_000, 128, 4_000, False), (250_000, 128, 20_000, False), (320_000, 128, 4_000, False),
                                         (156_000, 64, 20_000, False), (311_296, 128, 20_000, True), (311_296, 64, 2_048, True),
                                         (400_000, 64, 2_048, True), (100_000, 64, 2_048, False), (311_296, 64, 1_700, False)])
def test_rounds(geek, n, d, k, pairs):
    from torch.profiler import ProfilerActivity, profile

    g = torch.Generator(device="cuda").manual_seed(1)
    c = torch.rand(k, d, generator=g, device="cuda") * 20 - 10
    x = c[torch.randint(0, k, (n,), generator=g, device="cuda")] + torch.randn(n, d, generator=g, device="cuda")
    ctx = geek.Context(0)
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("rounds of 152 SMs")
    _assign(geek, ctx, x, c.double(), geek.PREC_BF16)
    for _ in range(2):  # the first profile of a process may see nothing
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            _assign(geek, ctx, x, c.double(), geek.PREC_BF16)
            torch.cuda.synchronize()
        names = " ".join(e.name for e in p.events())
    assert "k_assign_tc" in names
    assert ("k_assign_tc_pair" in names) == pairs
