"""What a user of this package has it do, as measurable cases.

Each case is one call path of the public Python API (``nnsemd.Context``,
``nnsemd.Proposal``, ``knn.EMDKNN``, ``colour_transfer.transfer``) on seeded
inputs shaped like the workloads of ``paper_2401_07378_gb300.workloads``.

families (the key "kind" of a case)
  pair       one pair of low-dimensional histograms (d <= 8), ``Context.solve``
  transfer   colour transfer between two images, quantisation to recolouring
  images     a batch of pixel-grid image pairs, ``Context.solve_batched``
  docs       one query document against a collection, ``EMDKNN.distances``
  retrieval  a batch of descriptor-signature pairs, ``Context.solve_batched``
  cloud      one pair of high-dimensional clouds (d > 8), ``Context.solve``
"""
import functools
import math
import random

import numpy as np
import torch

from paper_2401_07378_gb300 import colour_transfer, knn, nnsemd

PIXELS = 28  # side of the pixel grid of the image histograms


def listed():
    return [
        # the smallest call: one pair of spatial-location histograms, its distance only
        dict(name="pair_256", kind="pair", m=256, n=256, d=2, metric="l2", protocol="greedy", points="uniform",
             weights="uniform", plan=False),
        # a mid-size ragged colour histogram pair with its transport plan, served in a seeded random order
        dict(name="colour_20011_random", kind="pair", m=20011, n=20011, d=3, metric="sql2", protocol="random",
             points="colours", weights="uniform", plan=True),
        # the colour histograms of two whole 256 x 256 images, their distance only
        dict(name="colour_65536", kind="pair", m=65536, n=65536, d=3, metric="sql2", protocol="greedy",
             points="colours", weights="uniform", plan=False),
        # colour transfer as an application: a 512 x 512 image recoloured after another one
        dict(name="transfer_512x512", kind="transfer", source=262144, reference=262144, k=256, iters=8),
        # image classification / clustering: many pixel-grid histogram pairs at once
        dict(name="images_2048", kind="images", pairs=2048, lo=80, hi=400, d=2, metric="l2"),
        # document kNN in FP32, the classifier's default
        dict(name="docs_4096_fp32", kind="docs", docs=4096, d=300, median=60, metric="l2", precision="fp32"),
        # document kNN with BF16 distances
        dict(name="docs_4096_bf16", kind="docs", docs=4096, d=300, median=60, metric="l2", precision="bf16"),
        # image retrieval: a batch of descriptor signatures, FP16 distances, tuned launch shapes
        dict(name="retrieval_1000_fp16", kind="retrieval", pairs=1000, lo=256, hi=2048, d=128, metric="l2",
             precision="fp16"),
        # two descriptor sets compared on their own: latency counts
        dict(name="cloud_300x700_d128", kind="cloud", m=300, n=700, d=128, metric="l2", precision="fp32",
             rerank_k=0, learned=False, plan=False),
        # a mixture cloud in plain FP32
        dict(name="cloud_16384_fp32", kind="cloud", m=16384, n=16384, d=64, metric="l2", precision="fp32",
             rerank_k=0, learned=False, plan=True),
        # large mixture clouds on the tensor cores
        dict(name="cloud_131072_bf16x3", kind="cloud", m=131072, n=131072, d=64, metric="l2", precision="bf16x3",
             rerank_k=8, learned=False, plan=True),
        # the same with the learned candidate proposal
        dict(name="cloud_131072_learned", kind="cloud", m=131072, n=131072, d=64, metric="l2", precision="bf16x3",
             rerank_k=8, learned=True, plan=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["pair", "pair", "transfer", "images", "docs", "retrieval", "cloud", "cloud", "cloud"])
    if kind == "pair":
        points = rng.choice(["uniform", "colours"])
        m, n = _log_int(rng, 64, 65536), 0
        n = min(65536, max(16, int(m * math.exp(rng.uniform(-1.0, 1.0)))))
        d = 3 if points == "colours" else rng.choice([1, 2, 2, 3, 3, 4, 5, 8])
        return dict(kind="pair", m=m, n=n, d=d, metric=rng.choice(["l2", "sql2", "l1"]),
                    protocol=rng.choice(["greedy", "greedy", "random"]), points=points,
                    weights=rng.choice(["uniform", "dirichlet"]), plan=rng.random() < 0.5)
    if kind == "transfer":
        return dict(kind="transfer", source=_log_int(rng, 16384, 262144), reference=_log_int(rng, 16384, 262144),
                    k=_log_int(rng, 16, 256), iters=rng.randint(2, 8))
    if kind == "images":
        lo = rng.randint(30, 100)
        return dict(kind="images", pairs=_log_int(rng, 64, 2048), lo=lo, hi=rng.randint(lo + 50, 400), d=2,
                    metric=rng.choice(["l2", "sql2", "l1"]))
    if kind == "docs":
        return dict(kind="docs", docs=_log_int(rng, 128, 4096), d=rng.choice([32, 50, 100, 128, 200, 300]),
                    median=rng.randint(30, 90), metric=rng.choice(["l2", "sql2"]),
                    precision=rng.choice(["fp32", "fp32", "bf16", "fp16"]))
    if kind == "retrieval":
        precision = rng.choice(["fp32", "fp16", "fp16", "bf16"])
        lo = rng.choice([64, 100, 256])
        return dict(kind="retrieval", pairs=_log_int(rng, 50, 300 if precision == "fp32" else 1000), lo=lo,
                    hi=rng.randint(lo + 100, 2048), d=rng.choice([64, 96, 128]), metric=rng.choice(["l2", "sql2"]),
                    precision=precision)
    form = rng.choice(["small", "fp32", "fp32", "reduced", "learned"])
    if form == "small":
        return dict(kind="cloud", m=rng.randint(20, 1500), n=rng.randint(20, 1500),
                    d=rng.choice([16, 50, 64, 128, 300]), metric=rng.choice(["l2", "sql2", "l1"]), precision="fp32",
                    rerank_k=0, learned=False, plan=rng.random() < 0.3)
    if form == "fp32":
        m = _log_int(rng, 2048, 16384)
        return dict(kind="cloud", m=m, n=min(16384, int(m * rng.uniform(0.6, 1.6))),
                    d=rng.choice([9, 16, 30, 64, 100, 128]), metric=rng.choice(["l2", "sql2", "l1"]),
                    precision="fp32", rerank_k=0, learned=False, plan=True)
    m = _log_int(rng, 8192, 98304)
    n = min(98304, int(m * rng.uniform(0.7, 1.4)))
    if form == "reduced":
        return dict(kind="cloud", m=m, n=n, d=rng.choice([32, 50, 64, 100, 128]), metric=rng.choice(["l2", "sql2"]),
                    precision=rng.choice(["bf16x3", "bf16x3", "fp16"]), rerank_k=rng.choice([0, 8]),
                    learned=False, plan=True)
    return dict(kind="cloud", m=m, n=n, d=rng.choice([32, 64, 64]), metric=rng.choice(["l2", "sql2"]),
                precision=rng.choice(["bf16x3", "bf16x3", "fp32"]), rerank_k=8, learned=True, plan=True)


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _context():
    """One context per process, as a program keeps it."""
    return nnsemd.Context(torch.cuda.current_device())


def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * (seed + 1) + salt)
    return g


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _uniform(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda")


def _dirichlet(g, n):
    """Unnormalised Dirichlet(1) weights: Exp(1) draws."""
    return -torch.log1p(-torch.rand(n, generator=g, device="cuda", dtype=torch.float64))


def _colours(g, n, centres, sigma=0.08):
    """Colour clusters clipped to [0, 1), as the pixels of an image."""
    lab = torch.randint(0, centres.shape[0], (n,), generator=g, device="cuda")
    return (centres[lab] + sigma * _normal(g, n, 3)).clamp_(0.0, 1.0 - 2.0 ** -24).contiguous()


def _mixture(g, n, means):
    """Points of a Gaussian mixture (sigma 0.5) with Dirichlet(1/2) weights."""
    lab = torch.randint(0, means.shape[0], (n,), generator=g, device="cuda")
    pts = (means[lab] + 0.5 * _normal(g, n, means.shape[1])).contiguous()
    w = _normal(g, n).double().square() * 0.5 + 1e-30
    return pts, w


def _mixture_means(d):
    return 2.0 * _normal(_gen(12345, d), 256, d)


def _sizes(case, seed, salt):
    rng = random.Random(1000003 * (seed + 1) + salt)
    m = [rng.randint(case["lo"], case["hi"]) for _ in range(case["pairs"])]
    off = np.zeros(len(m) + 1, np.int64)
    off[1:] = np.cumsum(m)
    return off


def _pair_inputs(case, seed):
    g = _gen(seed, 1)
    m, n, d = case["m"], case["n"], case["d"]
    if case["points"] == "colours":
        centres = _uniform(g, 8, 3)
        x, y = _colours(g, m, centres), _colours(g, n, centres)
    else:
        x, y = _uniform(g, m, d), _uniform(g, n, d)
    if case["weights"] == "uniform":
        a = torch.ones(m, dtype=torch.float64, device="cuda")
        b = torch.ones(n, dtype=torch.float64, device="cuda")
    else:
        a, b = _dirichlet(g, m), _dirichlet(g, n)
    return x, a, y, b


def _transfer_inputs(case, seed):
    """Two images: the reference has other clusters and a flat share of colours."""
    g = _gen(seed, 2)
    src = _colours(g, case["source"], _uniform(g, 8, 3))
    ref = (0.6 * _colours(g, case["reference"], _uniform(g, 8, 3)) + 0.3 * _uniform(g, case["reference"], 3))
    return src, ref.clamp_(0.0, 1.0).contiguous()


def _images_inputs(case, seed):
    """Images as distinct pixels of a 28 x 28 grid with grey values 1..255."""
    g = _gen(seed, 3)
    sides = []
    for salt in (31, 32):
        off = _sizes(case, seed, salt)
        order = torch.rand(case["pairs"], PIXELS * PIXELS, generator=g, device="cuda").argsort(1)
        cnt = torch.as_tensor(np.diff(off), device="cuda")
        keep = torch.arange(PIXELS * PIXELS, device="cuda")[None, :] < cnt[:, None]
        pix = order[keep]
        pts = torch.stack([pix // PIXELS, pix % PIXELS], 1).float().contiguous()
        w = torch.randint(1, 256, (pts.shape[0],), generator=g, device="cuda").double()
        sides.append((pts, w, off))
    return sides


@functools.lru_cache(maxsize=2)
def _vocabulary(d, size=50000):
    v = _normal(_gen(77, d), size, d)
    v = (v / v.norm(dim=1, keepdim=True)).contiguous()
    p = torch.arange(1, size + 1, device="cuda", dtype=torch.float64) ** -1.1
    return v, torch.log(p / p.sum()).float(), p


def _docs_inputs(case, seed):
    """Documents of distinct words drawn ~ rank^-1.1 (Gumbel top-k), weights
    ~ rank^-1.1, lengths LogNormal(ln median, 0.6) clipped to [20, 500]; the
    last one is the query."""
    g = _gen(seed, 4)
    vocab, logp, term = _vocabulary(case["d"])
    count = case["docs"] + 1
    length = torch.exp(math.log(case["median"]) + 0.6 * _normal(g, count)).round().clamp(20, 500).long()
    ids = []
    for lo in range(0, count, 512):
        hi = min(count, lo + 512)
        u = torch.rand(hi - lo, vocab.shape[0], generator=g, device="cuda").clamp_(1e-12, 1.0 - 1e-7)
        top = (logp[None, :] - torch.log(-torch.log(u))).topk(int(length[lo:hi].max()), dim=1).indices
        keep = torch.arange(top.shape[1], device="cuda")[None, :] < length[lo:hi, None]
        ids.append(top[keep])
    ids = torch.cat(ids)
    off = np.zeros(count + 1, np.int64)
    off[1:] = np.cumsum(length.cpu().numpy())
    q = int(off[-2])
    return vocab[ids[:q]].contiguous(), term[ids[:q]].contiguous(), off[:-1], vocab[ids[q:]].contiguous(), \
        term[ids[q:]].contiguous()


def _retrieval_inputs(case, seed):
    g = _gen(seed, 5)
    sides = []
    for salt in (51, 52):
        off = _sizes(case, seed, salt)
        pts = _normal(g, int(off[-1]), case["d"]).abs_()
        pts = (pts * (512.0 / pts.norm(dim=1, keepdim=True))).contiguous()
        sides.append((pts, _dirichlet(g, int(off[-1])), off))
    return sides


def _cloud_inputs(case, seed):
    g = _gen(seed, 6)
    means = _mixture_means(case["d"])
    return _mixture(g, case["m"], means) + _mixture(g, case["n"], means)


def _proposal(ctx, d):
    """A proposal as a program keeps it: fitted and trained on other seeds."""
    means = _mixture_means(d)
    prop = nnsemd.Proposal(ctx, d, cells=4096, hidden=256, seed=7)
    prop.fit(_mixture(_gen(501, d), 65536, means)[0], iters=5, seed=7)
    ys, xs = [], []
    for s in range(16):
        x = _mixture(_gen(600 + s, d), 4096, means)[0]
        y = _mixture(_gen(700 + s, d), 4096, means)[0]
        ys.append(y)
        xs.append(x[ctx.nearest(x, y, "l2").long()])
    prop.train(torch.cat(ys).contiguous(), torch.cat(xs).contiguous(), epochs=4, batch=4096, lr=2e-3, seed=7)
    return prop


_INPUTS = dict(pair=_pair_inputs, transfer=_transfer_inputs, images=_images_inputs, docs=_docs_inputs,
               retrieval=_retrieval_inputs, cloud=_cloud_inputs)


def prepare(case, seed):
    ctx = _context()
    inputs = _INPUTS[case["kind"]](case, seed)
    state = dict(ctx=ctx, case=case, inputs=inputs)
    if case["kind"] == "docs":
        x, a, off, y, b = inputs
        state["knn"] = knn.EMDKNN(ctx, x, a, off, np.zeros(case["docs"], np.int64), metric=case["metric"],
                                  precision=case["precision"])
    if case.get("learned"):
        state["proposal"] = _proposal(ctx, case["d"])
    return state


def _plan_by_consumer(r, m):
    """The cost and the plan ordered by what each consumer receives (a plan's
    entries come in no fixed order)."""
    order = torch.argsort(r.plan_j.long() * m + r.plan_i)
    return {"cost": r.cost, "i": r.plan_i[order], "j": r.plan_j[order], "f": r.plan_f[order]}


def run(state):
    case, ctx, inputs = state["case"], state["ctx"], state["inputs"]
    kind = case["kind"]
    if kind == "pair":
        x, a, y, b = inputs
        r = ctx.solve(x, a, y, b, metric=case["metric"], plan=case["plan"], protocol=case["protocol"], seed=11)
        return _plan_by_consumer(r, case["m"]) if case["plan"] else {"cost": r.cost}
    if kind == "transfer":
        r = colour_transfer.transfer(ctx, inputs[0], inputs[1], k=case["k"], iters=case["iters"])
        return {"cost": r.cost, "pixels": r.pixels, "labels": r.labels, "source_palette": r.source_palette,
                "reference_palette": r.reference_palette, "mapped_palette": r.mapped_palette}
    if kind == "images":
        (x, a, xo), (y, b, yo) = inputs
        return ctx.solve_batched(x, a, xo, y, b, yo, metric=case["metric"])[0]
    if kind == "docs":
        return state["knn"].distances(inputs[3], inputs[4])
    if kind == "retrieval":
        (x, a, xo), (y, b, yo) = inputs
        flags = nnsemd.FLAG_AUTOTUNE if case["precision"] != "fp32" else 0
        return ctx.solve_batched(x, a, xo, y, b, yo, metric=case["metric"], precision=case["precision"],
                                 flags=flags)[0]
    x, a, y, b = inputs
    r = ctx.solve(x, a, y, b, metric=case["metric"], precision=case["precision"], rerank_k=case["rerank_k"],
                  plan=case["plan"], proposal=state.get("proposal"))
    return _plan_by_consumer(r, case["m"]) if case["plan"] else {"cost": r.cost}


# --------------------------------------------------------------------------
# work: inputs read once, outputs written once; the operations are those of
# one distance matrix where d > 8 leaves no way around it (the proposal's
# network and cell scores where it replaces the matrix), and of the cost terms
# --------------------------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind == "pair":
        m, n, d = case["m"], case["n"], case["d"]
        out = 8 + (16 * (m + n) if case["plan"] else 0)
        return {"bytes": (4 * d + 8) * (m + n) + out, "flops": 3 * d * (m + n)}
    if kind == "transfer":
        s, r, k = case["source"], case["reference"], case["k"]
        nearest = 3 * 3 * math.log2(max(2, k))  # a search tree over the palette
        return {"bytes": 12 * (s + r) + 16 * s, "flops": (s + r) * (case["iters"] + 1) * (nearest + 3)}
    if kind == "images":
        pts = case["pairs"] * (case["lo"] + case["hi"])
        return {"bytes": 16 * pts + 8 * case["pairs"], "flops": 3 * case["d"] * pts}
    if kind == "docs":
        mean = case["median"] * math.exp(0.18)
        words = case["docs"] * mean
        return {"bytes": (4 * case["d"] + 8) * (words + mean) + 8 * case["docs"],
                "flops": 2 * case["d"] * words * mean}
    if kind == "retrieval":
        mean = (case["lo"] + case["hi"]) / 2
        return {"bytes": (4 * case["d"] + 8) * 2 * mean * case["pairs"] + 8 * case["pairs"],
                "flops": 2 * case["d"] * mean * mean * case["pairs"]}
    m, n, d = case["m"], case["n"], case["d"]
    io = (4 * d + 8) * (m + n) + 8 + (16 * (m + n) if case["plan"] else 0)
    if case["learned"]:
        cells, hidden = 4096, 256
        return {"bytes": io, "flops": 2.0 * n * (d * hidden + hidden * hidden + hidden * cells) + 2.0 * m * d * cells}
    return {"bytes": io, "flops": 2.0 * m * n * d}


# --------------------------------------------------------------------------
# the same in 64 bits, without this package's solver
# --------------------------------------------------------------------------

def _dist_rows(x, y, metric):
    """[len(y), len(x)]: squared distances (L1 sums for l1) in 64 bits."""
    if metric == "l1":
        return torch.cdist(y, x, p=1.0)
    if x.shape[1] <= 8:
        d2 = torch.zeros(y.shape[0], x.shape[0], dtype=torch.float64, device=x.device)
        for k in range(x.shape[1]):
            d2 += (y[:, k, None] - x[None, :, k]).square_()
        return d2
    return torch.addmm((x * x).sum(1)[None, :], y, x.T, alpha=-2.0) + (y * y).sum(1)[:, None]


def _key64(x, y, metric):
    """Distance key of matching rows, by direct differences."""
    t = x - y
    return t.abs().sum(1) if metric == "l1" else t.square().sum(1)


def _nearest64(x, y, metric):
    """The nearest row of x for every row of y (the first one of equal keys)."""
    step = max(1, (1 << 26) // max(1, x.shape[0]))
    return torch.cat([_dist_rows(x, y[lo:lo + step], metric).argmin(1) for lo in range(0, y.shape[0], step)])


class _Padded:
    """Nearest suppliers inside each pair of a batch, from padded matrices."""

    def __init__(self, x, xo, y, yo, metric):
        xo, yo = torch.as_tensor(xo, device=x.device), torch.as_tensor(yo, device=x.device)
        mx, my = int((xo[1:] - xo[:-1]).max()), int((yo[1:] - yo[:-1]).max())
        self.xo, self.yo = xo, yo
        px, py = xo[:-1, None] + torch.arange(mx, device=x.device), yo[:-1, None] + torch.arange(my, device=x.device)
        bad = px >= xo[1:, None]
        px, py = px.clamp(max=x.shape[0] - 1), py.clamp(max=y.shape[0] - 1)
        dist = []
        step = max(1, (1 << 27) // (mx * my))
        for lo in range(0, px.shape[0], step):
            u, v = x[px[lo:lo + step]], y[py[lo:lo + step]]
            if metric == "l1":
                dist.append(torch.cdist(v, u, p=1.0))
            else:
                d2 = torch.baddbmm((u * u).sum(2)[:, None, :], v, u.transpose(1, 2), alpha=-2.0)
                dist.append(d2.add_((v * v).sum(2)[:, :, None]))
        self.dist = torch.cat(dist).masked_fill_(bad[:, None, :], math.inf)

    def pair_of(self, j):
        return torch.searchsorted(self.yo, j, right=True) - 1

    def nearest(self, i_act, j_act):
        live = torch.zeros(int(self.xo[-1]) + 1, dtype=torch.bool, device=i_act.device)
        live[i_act] = True
        at = self.xo[:-1, None] + torch.arange(self.dist.shape[2], device=live.device)
        dead = ~live[torch.minimum(at, self.xo[-1:, None])]
        p = self.dist.masked_fill_(dead[:, None, :], math.inf).argmin(2)
        pair = self.pair_of(j_act)
        i = p[pair, j_act - self.yo[pair]] + self.xo[pair]
        return i, live[i] & (i < self.xo[pair + 1])  # (a pair without active suppliers has none)


def _splitmix_key(seed, rnd, j):
    """Serving key of consumer j in a round: SplitMix64's output, upper half."""
    with np.errstate(over="ignore"):
        c = (np.uint64(rnd) << np.uint64(32)) | j.astype(np.uint64)
        z = np.uint64(seed) + (c + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z ^= z >> np.uint64(31)
    return (z >> np.uint64(32)).astype(np.int64)


def _flows64(nearest, x, s, y, c, metric, protocol="greedy", seed=0):
    """The rounds of NNS-EMD in 64 bits: the flows (i, j, f).  nearest(i_act,
    j_act) gives the nearest active supplier of each active consumer and
    whether there is one."""
    i_act, j_act = torch.nonzero(s > 0).flatten(), torch.nonzero(c > 0).flatten()
    fi, fj, ff = [], [], []
    rnd = 0
    while i_act.numel() and j_act.numel():
        i, there = nearest(i_act, j_act)
        if there is not None:
            i, j_act = i[there], j_act[there]
            if not j_act.numel():
                break
        if protocol == "random":
            key = torch.as_tensor(_splitmix_key(seed, rnd, j_act.cpu().numpy()), device=x.device)
        else:
            key = _key64(x[i], y[j_act], metric)
        order = torch.argsort(key, stable=True)
        order = order[torch.argsort(i[order], stable=True)]
        i, j = i[order], j_act[order]
        new = torch.ones_like(i, dtype=torch.bool)
        new[1:] = i[1:] != i[:-1]
        at = torch.nonzero(new).flatten()  # the next member of every group, served one each at a time
        end = torch.cat([at[1:], at.new_tensor([i.numel()])])
        while at.numel():
            ii, jj = i[at], j[at]
            si, cj = s[ii], c[jj]
            f = torch.minimum(si, cj)
            s[ii], c[jj] = si - f, cj - f
            fi.append(ii), fj.append(jj), ff.append(f)
            at = at + 1
            more = (at < end) & (s[ii] > 0)
            at, end = at[more], end[more]
        i_act, j_act = i_act[s[i_act] > 0], j_act[c[j_act] > 0]
        rnd += 1
    return torch.cat(fi), torch.cat(fj), torch.cat(ff)


def _terms64(x, y, fi, fj, ff, metric):
    return ff * (_key64(x[fi], y[fj], metric).sqrt() if metric == "l2" else _key64(x[fi], y[fj], metric))


def _solve64(x, a, y, b, metric, protocol="greedy", seed=0, flows=False):
    """NNS-EMD of one pair in 64 bits: the cost, and the flows if asked for."""
    x, y = x.double(), y.double()
    flow = _flows64(lambda i, j: (i[_nearest64(x[i], y[j], metric)], None), x, a / a.sum(), y, b / b.sum(), metric,
                    protocol, seed)
    cost = float(_terms64(x, y, *flow, metric).sum())
    return (cost,) + flow if flows else cost


def _solve64_batch(x, a, xo, y, b, yo, metric):
    """The costs of a packed batch of pairs in 64 bits."""
    x, y = x.double(), y.double()
    pad = _Padded(x, xo, y, yo, metric)

    def normalised(w, off):
        pair = torch.searchsorted(off, torch.arange(w.shape[0], device=w.device), right=True) - 1
        total = torch.zeros(off.shape[0] - 1, dtype=torch.float64, device=w.device).index_add_(0, pair, w)
        return w / total[pair]

    flow = _flows64(pad.nearest, x, normalised(a, pad.xo), y, normalised(b, pad.yo), metric)
    out = torch.zeros(pad.xo.shape[0] - 1, dtype=torch.float64, device=x.device)
    return out.index_add_(0, pad.pair_of(flow[1]), _terms64(x, y, *flow, metric))


def _kmeans64(pts, k, iters):
    pts = pts.double()
    n = pts.shape[0]
    cent = pts[((2 * torch.arange(k, device=pts.device) + 1) * n) // (2 * k)].clone()
    lab = _nearest64(cent, pts, "sql2")
    for _ in range(iters):
        cnt = torch.bincount(lab, minlength=k)
        mean = torch.zeros_like(cent).index_add_(0, lab, pts) / cnt.clamp(min=1)[:, None]
        cent = torch.where(cnt[:, None] > 0, mean, cent)
        lab = _nearest64(cent, pts, "sql2")
    return cent, lab, torch.bincount(lab, minlength=k)


def _transfer64(case, seed):
    src, ref = _transfer_inputs(case, seed)
    cs, ls, ns = _kmeans64(src, case["k"], case["iters"])
    cr, _, nr = _kmeans64(ref, case["k"], case["iters"])
    us, ur = ns > 0, nr > 0
    y, x = cs[us], cr[ur]
    cost, fi, fj, ff = _solve64(x, nr[ur].double(), y, ns[us].double(), "sql2", flows=True)
    num = torch.zeros_like(y).index_add_(0, fj, ff[:, None] * x[fi])
    den = torch.zeros(y.shape[0], dtype=torch.float64, device=y.device).index_add_(0, fj, ff)
    mapped = cs.clone()
    mapped[us] = torch.where(den[:, None] > 0, num / den[:, None], y)
    return {"cost": cost, "pixels": mapped[ls], "labels": None, "source_palette": cs, "reference_palette": cr,
            "mapped_palette": mapped}


def _exact_plan(case, cost):
    """(The plan's entries hang on each choice: only the cost is compared.)"""
    return {"cost": cost, "i": None, "j": None, "f": None} if case["plan"] else {"cost": cost}


def exact(case, seed):
    kind = case["kind"]
    if kind == "transfer":
        return _transfer64(case, seed)
    inputs = _INPUTS[kind](case, seed)
    if kind == "pair":
        cost = _solve64(*inputs, case["metric"], case["protocol"], 11)
        return _exact_plan(case, cost)
    if kind == "cloud":
        return _exact_plan(case, _solve64(*inputs, case["metric"]))
    if kind == "docs":  # the query once for every document
        x, a, off, y, b = inputs
        reps = case["docs"]
        return _solve64_batch(x, a, off, y.repeat(reps, 1), b.repeat(reps), np.arange(reps + 1) * y.shape[0],
                              case["metric"])
    (x, a, xo), (y, b, yo) = inputs
    return _solve64_batch(x, a, xo, y, b, yo, case["metric"])
