"""GPU: tables of many objects under keys of two words, sorted by the upper key
bits and then settled: runs of equal prefixes of 2 to some thousands of objects
whose lower bits differ, around the longest run of one thread (32) and a block's
step (2,048), at tile edges; tables of large buckets; and one-word keys beside
them.  The members must be the stable order of the codes."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2106_10515_gb300 import geek
    return geek


SMALL = [2] * 2000 + [3] * 500 + [31, 32, 33, 34, 65, 100, 200]


@pytest.mark.parametrize("n,L,w,sizes", [(540_001, 16, 1.5, SMALL), (540_001, 16, 0.1, []), (540_001, 16, 0.1, SMALL),
                                         (1_050_003, 8, 0.02, SMALL), (540_001, 16, 0.1, [2000] * 100),
                                         (24_000_003, 1, 0.01, [2047, 2048, 2049, 2100])])
def test_members_in_the_stable_order_of_the_codes(G, n, L, w, sizes):
    g = torch.Generator(device="cuda").manual_seed(n + L)
    K, d = 6, 4
    x = torch.randn(n, d, generator=g, device="cuda") * 100
    at = torch.randperm(n, generator=g, device="cuda")
    o = 0
    for s in sizes:  # equal in the coordinates of all functions but the last
        x[at[o:o + s], :3] = x[at[o], :3].clone()
        o += s
    if o:
        x[at[:o], 3] = torch.randint(0, 20, (o,), generator=g, device="cuda") * 2.5
    a = torch.randn(L, K, d, generator=g, device="cuda")
    a[:, :4, 2:] = 0
    a[:, 4, [0, 1, 3]] = 0
    a[:, 5, :3] = 0
    b = torch.rand(K * L, generator=g, device="cuda") * w
    ctx = G.Context(0)
    got = ctx.hash(ctx.dense(x), K, L, a=a.view(K * L, d).contiguous(), b=b, w=w).copy_out()
    codes = got["codes"].view(n, L, K).long()
    bits = 0
    for l in range(L):
        order = torch.arange(n, device="cuda")
        for k in reversed(range(K)):
            order = order[torch.sort(codes[order, l, k], stable=True).indices]
        assert torch.equal(got["members"].view(L, n)[l].long(), order)
        c = codes[order, l]
        start = torch.cat([torch.ones(1, dtype=torch.bool, device="cuda"), (c[1:] != c[:-1]).any(1)])
        rank = torch.empty(n, dtype=torch.long, device="cuda")
        rank[order] = torch.cumsum(start, 0) - 1
        assert torch.equal(got["obj_bucket"].view(L, n)[l].long(), rank)
        r = codes[:, l].amax(0) - codes[:, l].amin(0)
        bits = max(bits, sum(int(v).bit_length() for v in r.tolist()))
    assert (bits > 64) == (w < 0.5) and bits >= 49
