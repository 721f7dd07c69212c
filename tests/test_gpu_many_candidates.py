"""GPU: flagged rows with many candidates go to the FP32 scan of every centre:
labels around the line (64 candidates, a quarter and a sixth of the centres), in
both orders and in a batch, and what such a call costs."""
import time

import pytest
import torch

pytestmark = pytest.mark.gpu


def _points(n, d, k, off, apart, seed):
    """Points around k centres in groups of up to 40; off / apart decides how many are candidates."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    groups = max(1, k // 40)
    base = torch.randn(groups, d, generator=g, device="cuda") * 5 + off
    c = base[torch.arange(k, device="cuda") % groups] + torch.randn(k, d, generator=g, device="cuda") * apart
    x = base[torch.randint(0, groups, (n,), generator=g, device="cuda")] + torch.randn(n, d, generator=g, device="cuda") * 2 * apart
    return x, c.double()


def _labels(geek, ctx, x, c, prec):
    lab = torch.full((x.shape[0],), -7, dtype=torch.int32, device="cuda")
    return lab, ctx.assign_centers(ctx.dense(x), c, lab, precision=prec)


@pytest.mark.parametrize("prec", ["PREC_BF16", "PREC_BF16X3"])
@pytest.mark.parametrize("off", [3.0, 12.0, 40.0, 150.0, 600.0])
@pytest.mark.parametrize("n,d,k", [(700, 33, 63), (700, 64, 65), (900, 17, 257), (500, 100, 390), (130_001, 16, 65), (120_003, 32, 300)])
def test_labels_on_both_sides_of_the_line(geek, prec, off, n, d, k):
    x, c = _points(n, d, k, off, 0.5, n + k)
    ctx = geek.Context(0)
    want, _ = _labels(geek, ctx, x, c, geek.PREC_FP32)
    got, _ = _labels(geek, ctx, x, c, getattr(geek, prec))
    assert torch.equal(got, want)


def test_every_centre_a_candidate_costs_a_scan(geek):
    g = torch.Generator(device="cuda").manual_seed(5)
    n, d, k = 90_000, 128, 2_000
    c = torch.rand(k, d, generator=g, device="cuda") * 20 + 90  # far apart: FP32 decides every row
    x = c[torch.randint(0, k, (n,), generator=g, device="cuda")] + torch.randn(n, d, generator=g, device="cuda")
    c = c.double()
    ctx = geek.Context(0)

    def fastest(prec):
        t = []
        for _ in range(6):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            _, st = _labels(geek, ctx, x, c, prec)
            torch.cuda.synchronize()
            t.append(time.perf_counter() - t0)
        return min(t[1:]), st

    t32, _ = fastest(geek.PREC_FP32)
    t16, st = fastest(geek.PREC_BF16)
    assert st.n_recheck_rows == n and st.n_fp64_rows == 0
    # the same scan beside two tensor passes
    assert t16 < 3 * t32
