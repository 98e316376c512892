"""The workloads this library is timed on: graph builds, exact lists, graph
search and the inverted index that seeds it, each through the package's
public entry points.

A case is a dict of plain values.  "kind" names the entry point (build, plan,
batched, exact, search, train, index, seeds), "gen" the shape of the data:
  gmm    isotropic Gaussian mixture (centres U[-10, 10], sigma 1)
  sift   non-negative integers 0..255, clustered, about 30 % zeros
  gist   values in [0, 1], L1-normalised per block of 32 dims
  unit   unit-normalised Gaussian mixture
Inputs are drawn on the GPU from the seed alone.
"""
import math

import numpy as np
import torch

import paper_1701_08475_gb300 as knng

MASK = 2**64 - 1
PRECISION = {"fp32": knng.KNNG_FP32, "bf16": knng.KNNG_BF16, "fp16": knng.KNNG_FP16, "fp8": knng.KNNG_FP8}
JOIN = {"fwd": knng.KNNG_JOIN_FWD, "fwd_rev": knng.KNNG_JOIN_FWD_REV, "sampled": knng.KNNG_JOIN_SAMPLED}


def listed():
    return [
        # the smallest build: the plain FP32 form of the 10,000-point mixture, launches and host work count
        dict(name="build_gmm_10k", kind="build", gen="gmm", n=10_000, D=32, centres=50, k=10, leaf_max=64, passes=1,
             rounds=2, join="fwd_rev", precision="fp32", iters=4),
        # an ordinary build replayed from its recorded graph, as a service that rebuilds on new rows does
        dict(name="plan_sift_100k", kind="plan", gen="sift", n=100_003, D=128, centres=1000, k=20, leaf_max=128,
             passes=3, rounds=4, join="fwd_rev", precision="bf16", iters=4),
        # the headline workload: one million descriptors with integer values, called directly
        dict(name="build_sift_1m", kind="build", gen="sift", n=1_000_000, D=128, centres=1000, k=20, leaf_max=128,
             passes=3, rounds=4, join="fwd_rev", precision="bf16", iters=4),
        # wide rows with large leaves, values that 16 bits do not hold exactly
        dict(name="build_gist_100k", kind="build", gen="gist", n=100_000, D=960, centres=1000, k=20, leaf_max=256,
             passes=3, rounds=4, join="fwd_rev", precision="fp16", iters=4),
        # the largest: ten million unit vectors, FP8 leaves
        dict(name="build_unit_10m", kind="build", gen="unit", n=10_000_000, D=96, centres=10_000, k=16, leaf_max=128,
             passes=3, rounds=4, join="fwd_rev", precision="fp8", iters=4),
        # many independent graphs of uneven sizes and three dims in one call
        dict(name="batched_16", kind="batched", instances=16, n_lo=2_000, n_hi=100_000, k=16, leaf_max=128, passes=3,
             rounds=4, join="fwd_rev", precision="bf16", iters=4),
        # ground truth for the recall of a graph on a sample of its rows
        dict(name="exact_sift_1m", kind="exact", gen="sift", n=1_000_000, D=128, centres=1000, k=20, sample=2_000),
        # bulk search over a built graph
        dict(name="search_sift_1m", kind="search", gen="sift", n=1_000_000, D=128, centres=1000, k=20, m=10_000,
             s=32, t0=12, ks=20),
        # one online query
        dict(name="search_one", kind="search", gen="unit", n=100_000, D=96, centres=1000, k=16, m=1, s=32, t0=12,
             ks=10),
        # vocabularies of the inverted index from a prefix of the descriptors
        dict(name="train_sift_100k", kind="train", gen="sift", n=100_000, D=128, centres=1000, W1=256, W2=256,
             iters=8),
        # the whole input indexed with given vocabularies
        dict(name="index_sift_1m", kind="index", gen="sift", n=1_000_000, D=128, centres=1000, W1=256, W2=256),
        # seeds of a bulk search from the index
        dict(name="seeds_sift_10k", kind="seeds", gen="sift", n=300_000, D=128, centres=1000, W1=256, W2=256,
             m=10_000, probe1=16, s=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _rows(rng, D, lo, hi):
    """A number of rows, log-uniform, with at most 4e8 values in all."""
    return max(lo, min(_log(rng, lo, hi), int(4e8 / D)))


def _shape(rng):
    """Data and its dims: each recipe at its own dims and around them, odd ones too."""
    gen = rng.choice(["gmm", "sift", "gist", "unit"])
    if gen == "gist":
        return gen, 32 * rng.randint(4, 30)
    if gen == "sift":
        return gen, rng.choice([128, 128, 64, 100, 131])
    if gen == "unit":
        return gen, rng.choice([96, 96, 100, 200, 25])
    return gen, rng.choice([32, 64, 128, 256, rng.randint(8, 300)])


def draw(rng):
    kind = rng.choice(["build", "build", "plan", "build", "batched", "exact", "search", "search", "train", "index",
                       "seeds"])
    gen, D = _shape(rng)
    c = dict(kind=kind, gen=gen, D=D, centres=_log(rng, 50, 1000))
    if kind in ("build", "plan"):
        k = rng.choice([10, 16, 20])
        c.update(n=_rows(rng, D, 3_000, 2_000_000 if kind == "build" else 200_000), k=k,
                 leaf_max=rng.choice([64, 128, 256]), passes=rng.choice([1, 3]), rounds=rng.choice([0, 2, 4]),
                 join=rng.choice(["fwd_rev", "fwd_rev", "fwd"] + (["sampled"] if kind == "build" else [])),
                 precision=rng.choice(["fp32", "bf16", "fp16", "fp8"]), iters=rng.choice([2, 4]))
        if c["join"] == "sampled":
            c["rounds"] = max(2, c["rounds"])
    elif kind == "batched":
        c = dict(kind=kind, instances=rng.randint(2, 24), n_lo=2_000, n_hi=_log(rng, 4_000, 100_000), k=16,
                 leaf_max=rng.choice([64, 128, 256]), passes=3, rounds=4, join="fwd_rev",
                 precision=rng.choice(["fp32", "bf16"]), iters=rng.choice([2, 4]))
    elif kind == "exact":
        n = _rows(rng, D, 5_000, 1_000_000)
        c.update(n=n, k=rng.choice([10, 16, 20, 64]), sample=_log(rng, 100, min(2_000, n)))
    elif kind == "search":
        c.update(n=_rows(rng, D, 10_000, 1_000_000), k=rng.choice([10, 16, 20]), m=_log(rng, 1, 10_000),
                 s=rng.choice([16, 32, 40]), t0=rng.choice([6, 12]), ks=rng.choice([10, 20, 32]))
    elif kind == "train":
        W = rng.choice([64, 200, 256])
        c.update(n=min(_rows(rng, D, 5_000, 100_000), int(2.5e7 / D)), W1=W, W2=W, iters=rng.choice([4, 8]))
    elif kind == "index":
        c.update(n=_rows(rng, D, 5_000, 1_000_000), W1=rng.choice([64, 256]), W2=rng.choice([64, 200, 256]))
    else:
        c.update(n=_rows(rng, D, 10_000, 300_000), W1=256, W2=rng.choice([64, 256]), m=_log(rng, 1, 10_000),
                 probe1=rng.choice([8, 16, 32]), s=rng.choice([16, 32]))
    return c


# ---------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _uniform(shape, g, lo=0.0, hi=1.0):
    return torch.rand(shape, generator=g, device="cuda") * (hi - lo) + lo


def _normal(shape, g):
    return torch.randn(shape, generator=g, device="cuda")


def _data(gen, n, D, centres, seed):
    """n x D FP32 rows on the GPU."""
    g = _generator(seed)
    X = torch.empty((n, D), device="cuda")
    lab = torch.randint(0, centres, (n,), generator=g, device="cuda")
    if gen == "gmm":
        cen = _uniform((centres, D), g, -10.0, 10.0)
    elif gen == "sift":
        cen = _uniform((centres, D), g, 0.0, 120.0)
        keep = (_uniform((centres, D), g) >= 0.3).float()
        basis = _normal((centres, 16, D), g) * (25.0 / 4.0)
    elif gen == "gist":
        prof = torch._standard_gamma(torch.full((centres, D // 32, 32), 0.3, device="cuda"), generator=g) + 1e-3
        cen = (prof / prof.sum(2, keepdim=True)).reshape(centres, D)
    else:
        cen = _normal((centres, D), g)
        cen /= cen.norm(dim=1, keepdim=True)
    for a in range(0, n, 1 << 16):
        lb = lab[a:a + (1 << 16)]
        if gen == "gmm":
            v = _normal((len(lb), D), g) + cen[lb]
        elif gen == "sift":
            v = _normal((len(lb), D), g) * 4.0 + cen[lb]
            v += torch.bmm(_normal((len(lb), 1, 16), g), basis[lb]).squeeze(1)
            v = (v * keep[lb]).clamp_(0.0, 255.0).round_()
        elif gen == "gist":
            v = torch._standard_gamma(50.0 * cen[lb] + 1e-3, generator=g).reshape(len(lb), D // 32, 32)
            v = (v / v.sum(2, keepdim=True).clamp_min(1e-30)).reshape(len(lb), D)
        else:
            v = _normal((len(lb), D), g) * 0.1 + cen[lb]
            v /= v.norm(dim=1, keepdim=True)
        X[a:a + (1 << 16)] = v
    return X


def _params(c, seed):
    return knng.default_params(k=c["k"], leaf_max=c["leaf_max"], tree_passes=c["passes"], refine_rounds=c["rounds"],
                               join_mode=JOIN[c["join"]], precision=PRECISION[c["precision"]],
                               twomeans_iters=c["iters"], seed=seed, sample=c["k"] // 2 if c["join"] == "sampled" else 0)


def _batch_shapes(c):
    """The instances' (n, D, centres): uneven sizes spread over the case's range."""
    r = np.random.default_rng(c["instances"])
    at = (np.arange(c["instances"]) + r.random(c["instances"])) / c["instances"]
    return [(int(c["n_lo"] + t * (c["n_hi"] - c["n_lo"])), (64, 128, 256)[i % 3], int(r.integers(20, 501)))
            for i, t in enumerate(at)]


def _queries(X, gen, m, seed):
    """Rows of X moved by noise (rounded and clipped for integer rows), and which rows."""
    g = _generator(seed + 7919)
    base = torch.randint(0, X.shape[0], (m,), generator=g, device="cuda")
    sigma = {"gmm": 0.5, "sift": 4.0, "gist": 0.005, "unit": 0.05}[gen]
    Q = X[base] + _normal((m, X.shape[1]), g) * sigma
    if gen == "sift":
        Q = Q.clamp_(0.0, 255.0).round_()
    return Q.contiguous(), base, g


def _vocab(X, W1, W2, seed):
    """Two vocabularies with the values trained ones have: rows, and differences of rows of one neighbourhood."""
    g = _generator(seed + 104729)
    n = X.shape[0]
    w1 = X[torch.randperm(n, generator=g, device="cuda")[:W1]] * 0.875
    rows = X[torch.randperm(n, generator=g, device="cuda")[:W2]]
    near = torch.cdist(rows, w1).argmin(1)
    return w1.contiguous(), ((rows - w1[near]) * 0.75).contiguous()


def prepare(case, seed):
    c = dict(case)
    st = dict(case=c)
    if c["kind"] == "batched":
        st["data"] = [_data("gmm", n, D, cen, seed * 1000 + i) for i, (n, D, cen) in enumerate(_batch_shapes(c))]
        st["params"] = _params(c, seed)
        return st
    X = st["data"] = _data(c["gen"], c["n"], c["D"], c["centres"], seed)
    if c["kind"] == "build":
        st["params"] = _params(c, seed)
    elif c["kind"] == "plan":
        st["plan"] = knng.BuildPlan(X, _params(c, seed))
    elif c["kind"] == "exact":
        rows = np.sort(np.random.default_rng(seed).choice(c["n"], size=c["sample"], replace=False)).astype(np.int32)
        st["sample"] = torch.from_numpy(rows).cuda()
    elif c["kind"] == "search":
        # the graph a program has built before: three passes and two rounds
        p = knng.default_params(k=c["k"], leaf_max=128, tree_passes=3, refine_rounds=2, seed=seed)
        st["graph"] = knng.knng_build_ex(X, p)[0]
        st["queries"], base, g = _queries(X, c["gen"], c["m"], seed)
        S = torch.randint(0, c["n"], (c["m"], c["s"]), generator=g, device="cuda", dtype=torch.int32)
        S[:, 0] = st["graph"][base, -1]  # one seed near the query, as an index gives
        st["seeds"] = S
    elif c["kind"] == "index":
        st["words"] = _vocab(X, c["W1"], c["W2"], seed)
    elif c["kind"] == "seeds":
        w1, w2 = st["words"] = _vocab(X, c["W1"], c["W2"], seed)
        _, st["offsets"], st["lists"] = knng.knng_rvq_index(X, w1, w2)
        st["queries"] = _queries(X, c["gen"], c["m"], seed)[0]
    st["seed"] = seed
    return st


def run(st):
    c = st["case"]
    kind = c["kind"]
    if kind == "build":
        return knng.knng_build_ex(st["data"], st["params"])
    if kind == "plan":
        return st["plan"].launch()
    if kind == "batched":
        return knng.knng_build_batched(st["data"], st["params"])
    if kind == "exact":
        return knng.knng_exact(st["data"], c["k"], st["sample"])
    if kind == "search":
        return knng.knng_search(st["data"], st["graph"], st["queries"], st["seeds"], c["t0"], c["ks"])
    if kind == "train":
        return knng.knng_rvq_train(st["data"], c["W1"], c["W2"], c["iters"], seed=st["seed"])
    if kind == "index":
        return knng.knng_rvq_index(st["data"], *st["words"])
    return knng.knng_rvq_seeds(*st["words"], st["offsets"], st["lists"], st["queries"], c["probe1"], c["s"])


# ---------------------------------------------------------------- work
def _build_work(c, n, D):
    """The rows in and the lists out; the splits' projections and means, the leaves' pairs and the rounds' pairs
    (each node's members once with one another, of which most were compared before)."""
    leaf = c["leaf_max"] * 0.75
    levels = max(0, math.ceil(math.log2(max(1.0, n / c["leaf_max"]))))
    split = c["passes"] * levels * max(1, c["iters"]) * n * 3.0 * D
    leaves = c["passes"] * n * leaf / 2 * 2.0 * D
    join = c["rounds"] * n * (c["k"] * (c["k"] - 1) / 2) * 2.0 * D / 2
    return {"bytes": n * D * 4.0 + n * c["k"] * 8.0, "flops": split + leaves + join}


def work(case):
    c = case
    kind = c["kind"]
    if kind == "batched":
        each = [_build_work(c, n, D) for n, D, _ in _batch_shapes(c)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    n, D = c["n"], c["D"]
    if kind in ("build", "plan"):
        return _build_work(c, n, D)
    if kind == "exact":
        return {"bytes": n * D * 4.0 + c["sample"] * (4.0 + c["k"] * 8.0), "flops": 2.0 * c["sample"] * n * D}
    if kind == "search":
        # the call checks every row for non-finite values; about half of the slots offered are new rows
        visits = c["s"] + 0.5 * c["t0"] * c["ks"] * c["k"] / 4
        return {"bytes": n * D * 4.0 + c["m"] * (D * 4.0 + c["s"] * 4.0 + c["ks"] * 8.0),
                "flops": c["m"] * visits * 3.0 * D}
    if kind == "train":
        W = c["W1"] + c["W2"]
        return {"bytes": n * D * 4.0 + W * D * 4.0, "flops": 2.0 * n * D * (W * c["iters"] + c["W1"])}
    if kind == "index":
        return {"bytes": n * D * 4.0 + n * 12.0 + c["W1"] * c["W2"] * 4.0, "flops": 2.0 * n * D * (c["W1"] + c["W2"])}
    return {"bytes": c["m"] * (D * 4.0 + c["s"] * 4.0) + (c["W1"] + c["W2"]) * D * 4.0 + c["W1"] * c["W2"] * 4.0,
            "flops": 2.0 * c["m"] * (c["W1"] + c["W2"]) * D}


# ---------------------------------------------------------------- 64-bit values
def _exact_lists(c, st):
    """Squared distances of the k nearest rows, ascending, in 64 bits."""
    X, out = st["data"], []
    k = c["k"]
    for row in st["sample"].split(64):
        q = X[row.long()].double()
        best = torch.full((len(row), k), math.inf, dtype=torch.float64, device="cuda")
        for a in range(0, c["n"], 1 << 16):
            x = X[a:a + (1 << 16)].double()
            # |x|^2 + |q|^2 - 2 x.q chooses the rows, their difference gives the values
            part = (x * x).sum(1) + (q * q).sum(1, keepdim=True) - 2.0 * (q @ x.T)
            own = (row.long()[:, None] - a)
            inside = (own >= 0) & (own < x.shape[0])
            part.scatter_(1, own.clamp(0, x.shape[0] - 1), torch.where(inside, math.inf, part.gather(1, own.clamp(0, x.shape[0] - 1))))
            at = part.topk(min(k + 4, x.shape[0]), dim=1, largest=False)[1]
            d = ((x[at] - q[:, None]) ** 2).sum(2).masked_fill(part.gather(1, at).isinf(), math.inf)
            best = torch.cat([best, d], 1).sort(1)[0][:, :k]
        out.append(best)
    return torch.cat(out)


def _exact_search(c, st):
    """Alg. 2 in 64 bits: the rank list's first ks distances of every query."""
    X, G, ks, out = st["data"], st["graph"].long(), c["ks"], []
    big = c["n"]

    def first(q, ids, d, new):
        """The first ks distinct entries of (ids, d) and the ids `new`."""
        dn = torch.empty(new.shape, dtype=torch.float64, device="cuda")
        for b in range(0, new.shape[1], 64):
            dn[:, b:b + 64] = ((X[new[:, b:b + 64].clamp(0, big - 1)].double() - q[:, None]) ** 2).sum(2)
        dn = dn.masked_fill((new < 0) | (new >= big), math.inf)
        ids, d = torch.cat([ids, new], 1), torch.cat([d, dn], 1)
        o = ids.argsort(dim=1, stable=True)
        ids, d = ids.gather(1, o), d.gather(1, o)
        d[:, 1:] = d[:, 1:].masked_fill(ids[:, 1:] == ids[:, :-1], math.inf)
        o = d.argsort(dim=1, stable=True)[:, :ks]
        ids, d = ids.gather(1, o), d.gather(1, o)
        return ids.masked_fill(d.isinf(), -1), d

    for a in range(0, c["m"], 1000):
        q = st["queries"][a:a + 1000].double()
        none = torch.empty((len(q), 0), dtype=torch.int64, device="cuda")
        ids, d = first(q, none, none.double(), st["seeds"][a:a + 1000].long())
        for _ in range(c["t0"]):
            new = G[ids.clamp_min(0)].masked_fill((ids < 0)[:, :, None], -1).reshape(len(q), -1)
            ids, d = first(q, ids, d, new)
        out.append(torch.nn.functional.pad(d, (0, ks - d.shape[1]), value=math.inf))
    return torch.cat(out)


def _splitmix(z):
    z = (z + 0x9E3779B97F4A7C15) & MASK
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & MASK
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & MASK
    return z ^ (z >> 31)


def _lloyd(V, W, iters, seed, stage):
    """k-means from the stratified initial words; V in 64 bits."""
    n = V.shape[0]
    h = _splitmix((seed ^ (stage << 32)) & MASK)
    pos = []
    for w in range(W):
        lo, hi = w * n // W, (w + 1) * n // W
        pos.append(lo + _splitmix((h ^ w) & MASK) % (hi - lo))
    words = V[torch.tensor(pos, device="cuda")].clone()
    for _ in range(iters):
        code = _nearest(V, words)
        cnt = torch.bincount(code, minlength=W)
        mean = torch.zeros_like(words).index_add_(0, code, V) / cnt.clamp_min(1)[:, None]
        words = torch.where((cnt > 0)[:, None], mean, words)
    return words


def _nearest(V, words):
    out = []
    for v in V.split(1 << 16):
        out.append(((words * words).sum(1) - 2.0 * (v @ words.T)).argmin(1))
    return torch.cat(out)


def exact(case, seed):
    c = dict(case)
    # a build's distances follow its ids, and the index and the seeds are whole numbers
    if c["kind"] not in ("exact", "search", "train"):
        return None
    st = prepare(c, seed)
    if c["kind"] == "exact":
        return None, _exact_lists(c, st)
    if c["kind"] == "search":
        return None, _exact_search(c, st)
    V = st["data"].double()
    w1 = _lloyd(V, c["W1"], c["iters"], seed, 1)
    return w1, _lloyd(V - w1[_nearest(V, w1)], c["W2"], c["iters"], seed, 2)
