"""GPU: extra passes without room for the segments of large clusters sum them in one
chain each: the same centres and labels."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [60_000, (1 << 20) + 7])  # one stream; two
def test_without_segments(geek, n):
    g = torch.Generator(device="cuda").manual_seed(n)
    d, k = 20, 3
    c0 = torch.randn(k, d, generator=g, device="cuda") * 8
    lab0 = torch.randint(0, k, (n,), generator=g, device="cuda")
    x = c0[lab0] + torch.randn(n, d, generator=g, device="cuda")
    ctx = geek.Context(0)

    def refine():
        c, lab = c0.double(), lab0.int()
        ctx.refine(ctx.dense(x), c, lab, 1)  # FP32: no buffers of the tensor-core forms
        return c, lab

    want, went_on = refine(), 0
    for after in range(60):
        ctx.set_option(geek.OPT_TEST_FAIL_ALLOC, after)
        try:
            got = refine()
        except geek.GeekError as e:
            assert e.status == geek.ERR_NOMEM
            continue
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
        try:  # raises while the countdown still runs
            for _ in range(8):
                refine()
            went_on += 1
        except geek.GeekError as e:
            assert e.status == geek.ERR_NOMEM
        ctx.set_option(geek.OPT_TEST_FAIL_ALLOC, -1)
    assert went_on >= 2
