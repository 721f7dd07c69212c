"""GPU: a batch whose every row is flagged, instances of one row and of rows that
do not fill a warp among them: the rows are grouped by instance three times, and
every label must be that of the instance alone."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["PREC_BF16", "PREC_BF16X3"])
@pytest.mark.parametrize("off", [60.0, 2000.0])
def test_rows_of_many_instances(geek, prec, off):
    g = torch.Generator(device="cuda").manual_seed(9)
    u64 = lambda m: torch.randint(-(1 << 62), 1 << 62, (m,), generator=g, device="cuda", dtype=torch.int64)  # noqa: E731
    insts = []
    for i, n in enumerate((700, 1, 33, 3_000, 31, 32, 5_001, 64, 900)):
        d = (24, 64, 100)[i % 3]
        c = torch.randn(30, d, generator=g, device="cuda") * 4 + off
        x = c[torch.randint(0, 30, (n,), generator=g, device="cuda")] + torch.randn(n, d, generator=g, device="cuda")
        insts.append(dict(x=x, a=torch.randn(32, d, generator=g, device="cuda"), b=torch.rand(32, generator=g, device="cuda"),
                          w=4.0, mh_a=u64(60), mh_b=u64(60), dd_a=u64(3), dd_b=u64(3)))
    ctx = geek.Context(0)
    b = geek.Batch(ctx, insts, 4, 8, 3, 20, 2, precision=getattr(geek, prec))
    lab = torch.full((int(b.row_off[-1]),), -7, dtype=torch.int32, device="cuda")
    b.run(lab)
    out = b.copy_out()
    assert sum(o["k"] for o in out) > 0
    for i, I in enumerate(insts):
        got = lab[int(b.row_off[i]):int(b.row_off[i + 1])]
        if out[i]["k"] == 0:
            assert (got == -1).all()
            continue
        want = torch.empty_like(got)
        ctx.assign_centers(ctx.dense(I["x"]), geek._dev(out[i]["centres"]), want, precision=geek.PREC_FP32)
        assert torch.equal(got, want), i
