"""The workloads this framework's speed is measured on.

Every case is one call, or one chain of calls, a program makes through
paper_2106_10515_gb300.geek: hashing a data set into buckets, SILK seeding, the
one-pass assignment, extra passes of assignment, and the batch of many
instances.  Inputs are synthetic stand-ins of the paper's data sets (Gaussian
mixtures, Zipf item sets, heterogeneous rows), drawn on the GPU from a seed.

Kinds of cases and their fields (sizes of the listed ones are the
configurations of synth/, its parity cases, or ragged neighbours of them):

  assign  n x d points to k given centres        n, d, k, prec, stats
  refine  `passes` passes of update + assignment n, d, k, prec, passes
  hash    E2LSH / SRP codes and buckets          n, d, K, L, w, prec, srp
  dense   hash -> SILK -> centroids -> labels    n, d, comp, prec
  step    hash -> SILK -> labels of k centres    n, d, k, K, L
  alg1    Alg. 1 -> SILK -> centroids -> labels  n, d, comp, m, t, prec
  sets    MinHash -> SILK -> Jaccard labels      n, base, K, L, doph
  hetero  E2LSH ++ MinHash -> SILK -> modes      n, d, comp, K, L
  batch   `count` uneven instances in one plan   count, lo, hi
"""
import math

import numpy as np
import torch

from paper_2106_10515_gb300 import geek

PREC = {"fp32": geek.PREC_FP32, "bf16": geek.PREC_BF16, "bf16x3": geek.PREC_BF16X3}
UNIVERSE = 1 << 20  # items of the set data
# SILK decides the number of seeds; a program that keeps results of many runs
# side by side gives them buffers of one size, larger than any of its runs needs
MOST_SEEDS = {"raw": 1 << 14, "sets": 1 << 17, "doph": 1 << 14, "hetero": 1 << 14}
_ctx = None


def _context():
    """The one context a program creates and keeps."""
    global _ctx
    if _ctx is None:
        _ctx = geek.Context(torch.cuda.current_device())
    return _ctx


def listed():
    return [
        # a handful of new points labelled against existing clusters (serving): launches and latency
        dict(name="assign_few", kind="assign", n=777, d=32, k=50, prec="fp32", stats=False),
        # the small dense data set, whole pipeline with the default arithmetic
        dict(name="dense_20k", kind="dense", n=20_000, d=32, comp=50, prec="fp32"),
        # a mid-size labelling with a ragged dimension and centre count, split-BF16
        dict(name="assign_x3_300k", kind="assign", n=300_007, d=100, k=1_999, prec="bf16x3", stats=True),
        # the same with the default arithmetic of the call (FP32) on more rows
        dict(name="assign_fp32_1m", kind="assign", n=1_000_003, d=96, k=2_000, prec="fp32", stats=True),
        # hashing alone, default arithmetic, results copied out to the program
        dict(name="hash_2m", kind="hash", n=2_000_003, d=128, K=6, L=16, w=4.0, prec="fp32", srp=False),
        # the Sift10M-shaped step: hash, SILK and the assignment to the 20,000 mixture centres
        dict(name="step_10m", kind="step", n=10_000_000, d=128, k=20_000, K=6, L=16),
        # the paper's own dense pipeline (Alg. 1 even buckets, SILK decides k)
        dict(name="alg1_10m", kind="alg1", n=10_000_000, d=128, comp=20_000, m=40, t=5_000, prec="bf16x3"),
        # the URL-shaped sparse sets
        dict(name="sets_2m", kind="sets", n=2_000_000, base=5_000, K=4, L=32, doph=0),
        # the same kind of sets reduced by DOPH first
        dict(name="doph_500k", kind="sets", n=500_000, base=5_000, K=4, L=32, doph=400),
        # the GeoNames-shaped heterogeneous rows
        dict(name="hetero_2m", kind="hetero", n=2_000_000, d=20, comp=2_000, K=4, L=8),
        # many uneven instances clustered by one plan
        dict(name="batch_256", kind="batch", count=256, lo=10_000, hi=500_000),
        # Sect. 5's extra passes on the Sift10M-shaped points
        dict(name="refine_10m", kind="refine", n=10_000_000, d=128, k=20_000, prec="bf16", passes=2),
    ]


def _log_int(rng, lo, hi):
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, min(hi, v))


def draw(rng):
    kind = rng.choice(["assign", "assign", "refine", "hash", "dense", "step", "alg1", "sets", "doph", "hetero", "batch"])
    d = rng.choice([rng.randint(7, 128), 32, 64, 96, 100, 128])
    if kind == "assign":
        prec = rng.choice(["fp32", "bf16", "bf16x3"])
        n, k = _log_int(rng, 500, 10_000_000), _log_int(rng, 1, 20_000)
        most = 4e11 if prec == "fp32" else 1.2e13  # multiply-adds of a pass: below the largest listed case's time
        n = max(500, min(n, int(most / (k * d))))
        return dict(kind=kind, n=n, d=d, k=k, prec=prec, stats=rng.random() < 0.7)
    if kind == "refine":
        n = _log_int(rng, 5_000, 5_000_000)
        return dict(kind=kind, n=n, d=d, k=_log_int(rng, 20, min(20_000, n // 4)), prec=rng.choice(["bf16", "bf16x3"]), passes=rng.randint(1, 2))
    if kind == "hash":
        srp = rng.random() < 0.25
        K, L = (rng.randint(8, 16), rng.randint(4, 16)) if srp else (rng.randint(3, 6), rng.choice([8, 11, 16]))
        return dict(kind=kind, n=_log_int(rng, 1_000, 4_000_000), d=d, K=K, L=L, w=4.0, prec=rng.choice(["fp32", "bf16x3"]), srp=srp)
    if kind == "dense":
        return dict(kind=kind, n=_log_int(rng, 3_000, 200_000), d=rng.choice([20, 32, 64]), comp=rng.randint(20, 400), prec=rng.choice(["fp32", "bf16", "bf16x3"]))
    if kind == "step":
        return dict(kind=kind, n=_log_int(rng, 100_000, 10_000_000), d=rng.choice([64, 96, 100, 128]), k=_log_int(rng, 500, 20_000), K=rng.randint(4, 6), L=rng.choice([8, 16]))
    if kind == "alg1":
        n = _log_int(rng, 200_000, 5_000_000)
        return dict(kind=kind, n=n, d=rng.choice([64, 100, 128]), comp=max(50, n // 500), m=rng.choice([20, 40]), t=max(100, n // rng.randint(1_500, 2_500)), prec="bf16x3")
    if kind == "sets":
        n = _log_int(rng, 20_000, 1_500_000)
        return dict(kind=kind, n=n, base=max(50, n // 400), K=rng.choice([3, 4]), L=rng.choice([16, 32]), doph=0)
    if kind == "doph":
        n = _log_int(rng, 20_000, 400_000)
        return dict(kind="sets", n=n, base=max(50, n // 100), K=4, L=rng.choice([16, 32]), doph=rng.choice([64, 200, 400]))
    if kind == "hetero":
        return dict(kind=kind, n=_log_int(rng, 20_000, 2_000_000), d=rng.randint(8, 32), comp=rng.randint(100, 2_000), K=4, L=8)
    return dict(kind="batch", count=rng.randint(8, 160), lo=rng.choice([2_000, 10_000]), hi=rng.choice([100_000, 400_000]))


# ---- inputs ------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _u64(g, count):
    """Uniform 64-bit coefficients (the bits of a uint64 in an int64 tensor)."""
    return torch.randint(-(1 << 63), (1 << 63) - 1, (count,), generator=g, device="cuda", dtype=torch.int64)


def _silk(g, Ks, Ls, delta):
    return dict(Ks=Ks, Ls=Ls, delta=delta, mh_a=_u64(g, Ls * Ks), mh_b=_u64(g, Ls * Ks), dd_a=_u64(g, Ks), dd_b=_u64(g, Ks))


def _zipf(g, cdf, shape):
    """Ranks 0 .. len(cdf) - 1 by inverse CDF."""
    u = torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)
    return torch.searchsorted(cdf, u).clamp_(max=cdf.numel() - 1)


def _zipf_cdf(a, m):
    c = torch.arange(1, m + 1, device="cuda", dtype=torch.float64).pow_(-a).cumsum(0)
    return c / c[-1]


def _mixture(g, n, d, comp, reach=10.0, sigma=None, zipf=False):
    """Gaussian mixture: centres U[-reach, reach]^d; spread 1, or U[sigma] per
    component and dimension; equal or 1 / rank weights."""
    centres = (torch.rand((comp, d), generator=g, device="cuda") * 2 - 1) * reach
    if zipf:
        rank = _zipf(g, _zipf_cdf(1.0, comp), (n,))
        lab = torch.randperm(comp, generator=g, device="cuda")[rank]
    else:
        lab = torch.randint(0, comp, (n,), generator=g, device="cuda")
    x = torch.randn((n, d), generator=g, device="cuda")
    spread = None if sigma is None else sigma[0] + (sigma[1] - sigma[0]) * torch.rand((comp, d), generator=g, device="cuda")
    for s in range(0, n, 1 << 21):
        e = min(n, s + (1 << 21))
        if spread is not None:
            x[s:e] *= spread[lab[s:e]]
        x[s:e] += centres[lab[s:e]]
    return x, lab, centres


def _sift(g, n, d, comp):
    """Sift10M-shaped points: far centres, uneven spreads and weights."""
    return _mixture(g, n, d, comp, reach=50.0, sigma=(0.5, 2.0), zipf=True)


def _projection(g, F, d, w):
    a = torch.randn((F, d), generator=g, device="cuda")
    b = (torch.rand((F,), generator=g, device="cuda") * w).clamp_(max=float(np.nextafter(np.float32(w), np.float32(0))))
    return a, b


def _item_sets(g, n, base):
    """URL-shaped sets: 70 % of a set's Poisson(64) items from its cluster's base set, the rest Zipf(1.1) items."""
    cdf = _zipf_cdf(1.1, UNIVERSE)
    pois = lambda m: torch.poisson(torch.full((m,), 64.0, device="cuda"), generator=g).clamp_(min=1).long()  # noqa: E731
    far = 2 * UNIVERSE  # above every item
    b, _ = torch.sort(_zipf(g, cdf, (base, 512)), dim=1)
    b[:, 1:][b[:, 1:] == b[:, :-1]] = far
    # a random choice of each base set's distinct items
    key = torch.rand((base, 512), generator=g, device="cuda").masked_fill_(b == far, 2.0)
    order = key.argsort(dim=1)[:, :112]
    b = torch.gather(b, 1, order)
    size = torch.minimum(pois(base), (b != far).sum(1))
    col = torch.arange(112, device="cuda")
    counts, items = [], []
    for s in range(0, n, 250_000):
        m = min(250_000, n - s)
        lab = torch.randint(0, base, (m,), generator=g, device="cuda")
        want = pois(m)
        blen = size[lab]
        take = torch.minimum((0.7 * want).round().long(), blen)
        key = torch.rand((m, 112), generator=g, device="cuda").masked_fill_(col >= blen[:, None], 2.0)
        last = torch.gather(key.sort(dim=1).values, 1, (take - 1).clamp(min=0)[:, None])
        own = b[lab].masked_fill_((key > last) | (take == 0)[:, None], far)
        extra = _zipf(g, cdf, (m, 64)).masked_fill_(col[:64] >= (want - take)[:, None], far)
        row, _ = torch.sort(torch.cat([own, extra], 1), dim=1)
        keep = row < far
        keep[:, 1:] &= row[:, 1:] != row[:, :-1]
        counts.append(keep.sum(1))
        items.append(row[keep].to(torch.int32))
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cat(counts).cumsum(0)
    return off, torch.cat(items)


def _tokens(g, lab, comp, n_cat=10):
    """GeoNames-shaped categories: a home value per component, Zipf(1.2) steps from it; token = attribute offset + value."""
    card = [int(v) for v in torch.exp(math.log(10) + (math.log(1000) - math.log(10)) * torch.rand((n_cat,), generator=g, device="cuda")).tolist()]
    out = torch.empty((lab.numel(), n_cat), dtype=torch.int32, device="cuda")
    base = 0
    for j, c in enumerate(card):
        home = torch.randint(0, c, (comp,), generator=g, device="cuda")
        out[:, j] = ((home[lab] + _zipf(g, _zipf_cdf(1.2, c), (lab.numel(),))) % c + base).to(torch.int32)
        base += c
    return out


def _centre_rows(case):
    """Where the centroids go: room for more clusters than SILK finds on these data."""
    return torch.zeros((MOST_SEEDS["raw"], case["d"]), dtype=torch.float64, device="cuda")


def prepare(case, seed):
    g, ctx, kind = _gen(seed), _context(), case["kind"]
    s = dict(case=case, ctx=ctx)
    if kind in ("assign", "refine"):
        x, lab, c = _sift(g, case["n"], case["d"], case["k"])
        s.update(x=x, data=ctx.dense(x), centres=c.double(), labels=lab.to(torch.int32))
    elif kind in ("hash", "step"):
        w = case.get("w", 4.0)
        x, _, c = _sift(g, case["n"], case["d"], case.get("k", 2_000))
        a, b = _projection(g, case["K"] * case["L"], case["d"], w)
        s.update(x=x, data=ctx.dense(x), centres=c.double(), hash=dict(K=case["K"], L=case["L"], a=a, b=b, w=w), silk=_silk(g, 3, 10, 10))
    elif kind == "dense":
        x, _, _ = _mixture(g, case["n"], case["d"], case["comp"])
        a, b = _projection(g, 32, case["d"], 4.0)
        s.update(x=x, data=ctx.dense(x), hash=dict(K=4, L=8, a=a, b=b, w=4.0), silk=_silk(g, 3, 20, 2), centres=_centre_rows(case))
    elif kind == "alg1":
        x, _, _ = _sift(g, case["n"], case["d"], case["comp"])
        a, _ = _projection(g, case["m"], case["d"], 4.0)
        s.update(x=x, data=ctx.dense(x), hash=dict(K=1, L=case["m"], a=a, proj=geek.PROJ_QALSH, t=case["t"]), silk=_silk(g, 2, 20, 10), centres=_centre_rows(case))
    elif kind == "sets":
        off, items = _item_sets(g, case["n"], case["base"])
        F = case["K"] * case["L"]
        h = dict(K=case["K"], L=case["L"], mh_a=_u64(g, F), mh_b=_u64(g, F))
        if case["doph"]:
            p = [v & ((1 << 62) - 1) for v in _u64(g, 2).tolist()]
            h.update(doph_bins=case["doph"], doph_a=2 * p[0] + 1, doph_b=p[1])
        s.update(data=ctx.sets(off, items), hash=h, silk=_silk(g, 3, 20, 10))
    elif kind == "hetero":
        x, lab, _ = _mixture(g, case["n"], case["d"], case["comp"])
        tok = _tokens(g, lab, case["comp"])
        a, b = _projection(g, case["K"] * case["L"], case["d"], 4.0)
        h = dict(K=case["K"], L=case["L"], Kc=2, a=a, b=b, w=4.0, mh_a=_u64(g, 2 * case["L"]), mh_b=_u64(g, 2 * case["L"]))
        s.update(data=ctx.hetero(x, tok), hash=h, silk=_silk(g, 3, 20, 2))
    else:
        insts = []
        for n, d, comp in _batch_shapes(case):
            x, _, _ = _mixture(g, n, d, comp)
            a, b = _projection(g, 32, d, 4.0)
            sp = _silk(g, 3, 20, 2)
            insts.append(dict(x=x, a=a, b=b, w=4.0, mh_a=sp["mh_a"], mh_b=sp["mh_b"], dd_a=sp["dd_a"], dd_b=sp["dd_b"]))
        s.update(batch=geek.Batch(ctx, insts, 4, 8, 3, 20, 2), n=sum(i["x"].shape[0] for i in insts))
    return s


def _batch_shapes(case):
    """(n, d, components) of each instance: the shapes belong to the case, the values to the seed."""
    r = np.random.default_rng(2106105155)
    c = case["count"]
    n = np.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"]), c)).astype(int)
    return list(zip(n.tolist(), r.choice([32, 64, 128], c).tolist(), r.integers(10, 2001, c).tolist()))


# ---- one pass ------------------------------------------------------------------
def _labels(n):
    return torch.empty(n, dtype=torch.int32, device="cuda")


def _sized(t, rows):
    """t in a buffer of `rows` rows (more, if it has more), zeros behind it."""
    out = t.new_zeros((max(rows, t.shape[0]),) + tuple(t.shape[1:]))
    out[: t.shape[0]] = t
    return out


def _seeds(seeds, n, most):
    off, ids = seeds.copy_out()
    return dict(k=seeds.k, seed_off=_sized(off, most + 1), seed_ids=_sized(ids, 2 * n))


def run(s):
    case, ctx, kind = s["case"], s["ctx"], s["case"]["kind"]
    if kind == "assign":
        lab = _labels(case["n"])
        st = ctx.assign_centers(s["data"], s["centres"], lab, precision=PREC[case["prec"]], stats=case["stats"])
        return dict(labels=lab, sse=st.sse, radius=st.radius_max) if case["stats"] else dict(labels=lab)
    if kind == "refine":
        c, lab = s["centres"].clone(), s["labels"].clone()
        st = ctx.refine(s["data"], c, lab, case["passes"], precision=PREC[case["prec"]])
        return dict(labels=lab, centres=c, sse=st.sse, radius=st.radius_max)
    if kind == "hash":
        bk = ctx.hash(s["data"], precision=PREC[case["prec"]], proj=geek.PROJ_SRP if case["srp"] else geek.PROJ_E2LSH, **s["hash"])
        out = bk.copy_out()
        # the bucket offsets' length is the data's; obj_bucket, members and the counts determine them
        return {name: out[name] for name in ("obj_bucket", "n_buckets", "members", "codes")}
    if kind == "batch":
        lab = _labels(s["n"])
        s["batch"].run(lab)
        st = s["batch"].instance_stats()
        return dict(labels=lab, k=st["k"], sse=st["sse"], radius=st["radius_max"])
    if kind == "step":
        bk = ctx.hash(s["data"], precision=geek.PREC_BF16X3, **s["hash"])
        seeds = ctx.silk(bk, **s["silk"])
        lab = _labels(case["n"])
        st = ctx.assign_centers(s["data"], s["centres"], lab, precision=geek.PREC_BF16)
        return dict(labels=lab, n_buckets=bk.n_buckets, sse=st.sse, radius=st.radius_max, **_seeds(seeds, case["n"], MOST_SEEDS["raw"]))
    bk = ctx.hash(s["data"], **s["hash"])
    seeds = ctx.silk(bk, **s["silk"])
    lab = _labels(case["n"])
    if kind in ("dense", "alg1"):
        c = s["centres"]
        if seeds.k > c.shape[0]:
            c = torch.empty((seeds.k, case["d"]), dtype=torch.float64, device="cuda")
        st = ctx.assign(s["data"], bk, seeds, lab, centers=c, precision=PREC[case["prec"]])
        return dict(labels=lab, centres=c, sse=st.sse, radius=st.radius_max, **_seeds(seeds, case["n"], MOST_SEEDS["raw"]))
    st, cen = ctx.assign_ex(s["data"], bk, seeds, lab)
    if kind == "hetero":
        return dict(labels=lab, modes=_sized(cen["modes"], MOST_SEEDS[kind]), sse=st.sse, radius=st.radius_max, **_seeds(seeds, case["n"], MOST_SEEDS[kind]))
    if case["doph"]:
        return dict(labels=lab, modes=_sized(cen["modes"], MOST_SEEDS["doph"]), **_seeds(seeds, case["n"], MOST_SEEDS["doph"]))
    return dict(labels=lab, item_off=_sized(cen["item_off"], MOST_SEEDS["sets"] + 1), items=_sized(cen["items"], 1 << 24), **_seeds(seeds, case["n"], MOST_SEEDS["sets"]))


def work(case):
    """Bytes of the inputs and outputs and operations no form of the path can
    leave out (products of the projections and distances, hash evaluations).
    The pipelines' seed counts and bucket counts come from the data, so their
    centres, distances and bucket offsets are left out."""
    kind = case["kind"]
    if kind == "batch":
        sh = _batch_shapes(case)
        return dict(bytes=sum(4.0 * n * (d + 1) for n, d, _ in sh), flops=sum(64.0 * n * d for n, d, _ in sh))
    n = float(case["n"])
    if kind == "assign":
        return dict(bytes=4 * n * (case["d"] + 1) + 8.0 * case["k"] * case["d"], flops=2 * n * case["k"] * case["d"])
    if kind == "refine":
        kd = float(case["k"]) * case["d"]
        return dict(bytes=4 * n * (case["d"] + 2) + 16 * kd, flops=case["passes"] * (2 * n * kd + n * case["d"]))
    if kind == "sets":
        F = case["K"] * case["L"]
        items = case["doph"] if case["doph"] else 59  # mean items of a set, or its tokens
        out = 4 * n
        return dict(bytes=n * (8 + 4 * 59) + out, flops=2 * n * items * F)
    if kind == "alg1":
        return dict(bytes=4 * n * (case["d"] + 1), flops=2 * n * case["d"] * case["m"])
    if kind == "dense":
        return dict(bytes=4 * n * (case["d"] + 1), flops=64 * n * case["d"])
    F = case["K"] * case["L"]
    if kind == "hetero":
        return dict(bytes=4 * n * (case["d"] + 11), flops=2 * n * case["d"] * F + 40 * n * case["L"])
    if kind == "step":
        return dict(bytes=4 * n * (case["d"] + 1) + 8.0 * case["k"] * case["d"], flops=2 * n * case["d"] * (F + case["k"]))
    # hash: codes, bucket ids and members written
    return dict(bytes=4 * n * case["d"] + 4.0 * F * case["d"] + 4 * n * F + 8 * n * case["L"], flops=2 * n * case["d"] * F)


# ---- the same in 64 bits ---------------------------------------------------------
def _nearest(x, c):
    """Index of and 64-bit squared distance to each row's nearest centre: the two nearest in 32 bits, decided in 64."""
    n, k = x.shape[0], c.shape[0]
    c32, cn = c.float(), (c * c).sum(1).float()
    lab = torch.empty(n, dtype=torch.int64, device="cuda")
    dist = torch.empty(n, dtype=torch.float64, device="cuda")
    step = max(1, int(4e8) // max(k, x.shape[1]))
    allow = torch.backends.cuda.matmul.allow_tf32
    torch.backends.cuda.matmul.allow_tf32 = False
    for s in range(0, n, step):
        xs = x[s:s + step]
        v = torch.addmm(cn, xs, c32.t(), alpha=-2.0)
        x64 = xs.double()
        i1 = v.argmin(1)
        d1 = (x64 - c[i1]).square_().sum(1)
        if k > 1:
            v.scatter_(1, i1[:, None], float("inf"))
            i2 = v.argmin(1)
            d2 = (x64 - c[i2]).square_().sum(1)
            i1, d1 = torch.where(d2 < d1, i2, i1), torch.minimum(d1, d2)
        lab[s:s + step], dist[s:s + step] = i1, d1
    torch.backends.cuda.matmul.allow_tf32 = allow
    return lab, dist


def _means(x, lab, c):
    """64-bit means of the rows of each label; a centre without rows stays."""
    s = torch.zeros_like(c)
    for i in range(0, x.shape[0], 1 << 20):
        s.index_add_(0, lab[i:i + (1 << 20)], x[i:i + (1 << 20)].double())
    m = torch.bincount(lab, minlength=c.shape[0])[:, None]
    return torch.where(m > 0, s / m.clamp(min=1), c)


def exact(case, seed):
    """Labels, codes and seeds are whole numbers.  Distances and means are
    given where the centres are; where SILK chooses the seeds there is no
    plain form of the chain."""
    kind = case["kind"]
    if kind not in ("assign", "refine", "step") or (kind == "assign" and not case["stats"]):
        return None
    s = prepare(case, seed)
    x, c = s["x"], s["centres"]
    out = dict(labels=None)
    if kind == "refine":
        lab = s["labels"].long()
        for i in range(case["passes"]):
            c = _means(x, lab, c)
            lab, dist = _nearest(x, c)
        out["centres"] = c
    else:
        _, dist = _nearest(x, c)
    if kind == "step":
        out.update(k=None, seed_off=None, seed_ids=None, n_buckets=None)
    out.update(sse=float(dist.sum()), radius=float(dist.max().sqrt()))
    return out
