"""GPU: the buffer of the flagged rows' candidates stays within 1 GB however many
centres there are, and a call that cannot have all of it goes on with less."""
import ctypes as C

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

USED_CURRENT, USED_HIGH = 7, 8  # CU_MEMPOOL_ATTR_USED_MEM_*


def _pool():
    """(get, set) of an attribute of the device's default memory pool, which the library allocates from."""
    cu = C.CDLL("libcuda.so.1")
    pool = C.c_void_p()
    assert cu.cuDeviceGetDefaultMemPool(C.byref(pool), 0) == 0

    def get(a):
        v = C.c_uint64()
        assert cu.cuMemPoolGetAttribute(pool, a, C.byref(v)) == 0
        return v.value

    return get, lambda a: cu.cuMemPoolSetAttribute(pool, a, C.byref(C.c_uint64(0)))


def test_a_million_centres(geek):
    g = torch.Generator(device="cuda").manual_seed(1)
    n, d, k = 20_000, 8, 1_000_000
    c = torch.randn(k, d, generator=g, device="cuda", dtype=torch.float64) * 10
    x = torch.randn(n, d, generator=g, device="cuda") * 10
    ctx = geek.Context(0)
    want, got = (torch.empty(n, dtype=torch.int32, device="cuda") for _ in range(2))
    ctx.assign_centers(ctx.dense(x), c, want, precision=geek.PREC_FP32)
    torch.cuda.synchronize()
    get, reset = _pool()
    before = get(USED_CURRENT)
    assert reset(USED_HIGH) == 0
    st = ctx.assign_centers(ctx.dense(x), c, got, precision=geek.PREC_BF16)
    assert torch.equal(got, want)
    assert st.n_recheck_rows > 152 * 128  # more than a unit of 128 rows per SM
    # the centres in BF16, |c|^2 columns and FP32 parts: 300 MB
    assert get(USED_HIGH) - before < (1 << 30) + 400_000_000


def test_a_smaller_buffer_will_do(geek):
    g = torch.Generator(device="cuda").manual_seed(2)
    n, d, k = 4_000, 24, 300
    c = torch.randn(k, d, generator=g, device="cuda", dtype=torch.float64)
    x = torch.randn(n, d, generator=g, device="cuda")
    ctx = geek.Context(0)

    def assign(p):
        lab = torch.full((n,), -7, dtype=torch.int32, device="cuda")
        ctx.assign_centers(ctx.dense(x), c, lab, precision=p)
        return lab

    want, went_on = assign(geek.PREC_FP32), 0
    for after in range(60):
        ctx.set_option(geek.OPT_TEST_FAIL_ALLOC, after)
        try:
            got = assign(geek.PREC_BF16)
        except geek.GeekError as e:
            assert e.status == geek.ERR_NOMEM
            continue
        assert torch.equal(got, want)
        # the countdown is over: that allocation failed and the call went on
        try:
            for _ in range(60):
                assign(geek.PREC_FP32)
            went_on += 1
        except geek.GeekError as e:
            assert e.status == geek.ERR_NOMEM
        ctx.set_option(geek.OPT_TEST_FAIL_ALLOC, -1)
    assert went_on >= 1


def test_a_batch_goes_on_with_less(geek):
    g = torch.Generator(device="cuda").manual_seed(3)
    u64 = lambda m: torch.randint(-(1 << 62), 1 << 62, (m,), generator=g, device="cuda", dtype=torch.int64)  # noqa: E731
    insts = []
    for n, d in ((3_000, 16), (5_000, 80)):
        c = torch.randn(40, d, generator=g, device="cuda") * 8
        x = c[torch.randint(0, 40, (n,), generator=g, device="cuda")] + torch.randn(n, d, generator=g, device="cuda")
        insts.append(dict(x=x, a=torch.randn(32, d, generator=g, device="cuda"), b=torch.rand(32, generator=g, device="cuda"),
                          w=4.0, mh_a=u64(60), mh_b=u64(60), dd_a=u64(3), dd_b=u64(3)))

    def run(after):
        ctx = geek.Context(0)
        b = geek.Batch(ctx, insts, 4, 8, 3, 20, 2, precision=geek.PREC_BF16)
        ctx.set_option(geek.OPT_TEST_FAIL_ALLOC, after)
        lab = torch.full((8_000,), -7, dtype=torch.int32, device="cuda")
        try:
            b.run(lab)
        except geek.GeekError as e:
            assert e.status == geek.ERR_NOMEM
            return None, False
        try:  # raises while the countdown still runs
            ctx.assign_centers(ctx.dense(insts[0]["x"]), torch.zeros(2, 16, dtype=torch.float64, device="cuda"),
                               torch.empty(3_000, dtype=torch.int32, device="cuda"))
            over = True
        except geek.GeekError:
            over = False
        return lab, over

    want, _ = run(-1)
    assert want is not None and int(want.max()) > 0
    went_on = 0
    for after in range(400):
        got, over = run(after)
        if got is None:
            continue
        assert torch.equal(got, want)
        if not over:
            break
        went_on += 1
    assert went_on >= 1
