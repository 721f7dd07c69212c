"""GPU: Alg. 1 on data far from the origin: the parts are the oracle's whatever the
objects that give a table's middle value are, and the cost is that of centred data."""
import time

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["far", "farther", "two_sides", "outliers_in_the_middle", "huge", "one_value", "far_zeros"])
@pytest.mark.parametrize("n,t", [(31, 7), (777, 100), (5121, 60), (40_001, 350)])
def test_parts_equal_the_exact_split(geek, kind, n, t):
    rng = np.random.default_rng(n + len(kind))
    d, m = 9, 5
    x = rng.standard_normal((n, d))
    if kind == "far":
        x += 300
    elif kind == "farther":
        x += 1e6
    elif kind == "two_sides":
        x += 1e4 * rng.choice([-1, 1], (n, 1))
    elif kind == "outliers_in_the_middle":  # where a sample spread over the ids looks
        x[np.arange(31) * (n - 1) // 30] += 1e7
    elif kind == "huge":
        x *= 1e17
    elif kind == "one_value":
        x[:] = x[0] + 500
    elif kind == "far_zeros":
        x += 200
        x[rng.random(n) < 0.6] = 0
    x = x.astype(np.float32)
    a = rng.standard_normal((m, d)).astype(np.float32)
    ctx = geek.Context(0)
    got = ctx.hash(ctx.dense(geek._dev(x)), 1, m, a=geek._dev(a), proj=geek.PROJ_QALSH, t=t).copy_out()
    _, ref = oracle.transform_alg1(x, a, t)
    for key, r in (("obj_bucket", ref.obj_bucket), ("bucket_off", ref.boff), ("members", ref.bmem)):
        assert np.array_equal(got[key].cpu().numpy(), r), key


def test_distance_from_the_origin_costs_nothing(geek):
    g = torch.Generator(device="cuda").manual_seed(4)
    n, d, m, t = 1_000_000, 128, 20, 500
    x0 = torch.randn(n, d, generator=g, device="cuda") * 6
    a = torch.randn(m, d, generator=g, device="cuda")
    ctx = geek.Context(0)

    def fastest(off):
        data, s = ctx.dense(x0 + off), []
        for _ in range(6):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            ctx.hash(data, 1, m, a=a, proj=geek.PROJ_QALSH, t=t)
            torch.cuda.synchronize()
            s.append(time.perf_counter() - t0)
        return min(s[1:])

    # twice the time where FP32 values were rounded at their distance from the origin
    assert fastest(10_000.0) < 1.5 * fastest(0.0)
