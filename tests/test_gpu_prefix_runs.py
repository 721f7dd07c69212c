"""GPU: one long run of equal upper key bits among tables without any: the table
sort takes all its passes instead of leaving the run to one block; the order is the
stable one either way."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _passes(geek, n, L, one_run):
    """Radix passes of the table sort of n objects in L tables of six functions, one
    table's first five constant if one_run; and whether its members are in order."""
    g = torch.Generator(device="cuda").manual_seed(n + L)
    K, d, w = 6, 8, 0.05
    x = torch.randn(n, d, generator=g, device="cuda") * 100
    a = torch.randn(L, K, d, generator=g, device="cuda")
    if one_run:
        x[:, 0] = 0
        a[3, :K - 1, 1:] = 0  # see nothing of x
    b = torch.rand(K * L, generator=g, device="cuda") * w
    ctx = geek.Context(0)
    ctx.timing(True)
    bk = ctx.hash(ctx.dense(x), K, L, a=a.view(K * L, d).contiguous(), b=b, w=w)
    passes = ctx.timing_get("kernel.rs_scatter")[1]
    out = bk.copy_out()
    codes = out["codes"].view(n, L, K).long()
    for l in (0, 3, L - 1):
        order = torch.arange(n, device="cuda")
        for k in reversed(range(K)):
            order = order[torch.sort(codes[order, l, k], stable=True).indices]
        assert torch.equal(out["members"].view(L, n)[l].long(), order)
    return passes, bk.key_bits_max


@pytest.mark.parametrize("n,L", [(131_072, 64), (140_000, 60)])
def test_a_table_that_is_one_run_takes_every_pass(geek, n, L):
    passes, bits = _passes(geek, n, L, False)
    assert bits > 64 and passes <= (bits + 7) // 8 - 3  # upper bits alone
    passes, bits = _passes(geek, n, L, True)
    assert bits > 64 and passes == (bits + 7) // 8
