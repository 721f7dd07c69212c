"""GPU: the centre update of clusters large enough to be summed in parallel
segments equals the sequential FP64 chain bit for bit: values around a mean,
around zero, exact ties of the rounding, mixed exponents, cancelling and
vanishing sums, and cluster sizes around the segment and cluster limits."""
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


def _columns(rng, n):
    """Columns of float32 values, each a different way for the sum to round."""
    z = rng.standard_normal(n)
    cols = [30 + 2 * z, z, 0.3 + z, -17 + z, 1e-3 + z,
            np.ldexp(rng.integers(1, 1 << 24, n).astype(float), -20),       # many low bits
            np.ldexp(rng.integers(-(1 << 23), 1 << 23, n) * 2.0 + 1, -44) + 0.0,  # odd multiples: ties once s is large
            np.where(rng.random(n) < 0.5, 1.0, np.ldexp(1.0, -34)),         # exact halves of the sum's unit
            np.where(rng.random(n) < 0.5, 4096.0, -np.ldexp(3.0, -27)),
            z * np.exp2(rng.integers(-40, 20, n)),                          # mixed exponents
            np.where(np.arange(n) % 2, 5.0, -5.0) + 0.0,                    # returns to zero
            np.zeros(n), -np.zeros(n), np.full(n, 1e-42), z * 1e36,
            np.where(np.arange(n) == n // 3, 1e20, z),                      # one value dwarfs the rest
            np.where(np.arange(n) < n // 2, 1.0, -1.0) * 7 + z * 1e-3]      # grows, then falls back
    return np.stack(cols, 1).astype(np.float32)


@pytest.mark.parametrize("d,ldx", [(17, 17), (64, 68), (33, 40)])
def test_large_clusters_equal_the_sequential_sum(G, d, ldx):
    rng = np.random.default_rng(d)
    sizes = [40_000, 16_384, 16_385, 16_385 + 127, 20_480, 300, 0, 33_001]
    lab = np.repeat(np.arange(len(sizes)), sizes)
    lab = rng.permutation(np.concatenate([lab, np.full(200, -1)])).astype(np.int32)
    n = lab.size
    base = _columns(rng, n)
    x = np.zeros((n, ldx), np.float32)
    x[:, :d] = base[:, np.arange(d) % base.shape[1]]
    c0 = rng.standard_normal((len(sizes), d))
    ctx = G.Context(0)
    xd = G._dev(x)[:, :d]
    c, labels = G._dev(c0), G._dev(lab)
    ctx.refine(ctx.dense(xd), c, labels, 1, stats=False)
    torch.cuda.synchronize()
    got = c.cpu().numpy()
    for j, m in enumerate(sizes):
        rows = x[lab == j][:, :d].astype(np.float64)
        want = np.cumsum(rows, axis=0)[-1] / m if m else c0[j]
        assert np.array_equal(got[j], want), (j, np.flatnonzero(got[j] != want))
