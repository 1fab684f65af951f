"""What a user of this library has it do, as measurable cases.

A case is a dict of plain values; ``kind`` says which call sequence it stands
for:

* ``graph``    -- build a forest over a point matrix and take its kNN graph
  (``mode`` 0 plain float32, 1 BF16 Gram, 2 FP8 Gram);
* ``build``    -- build a forest and read every tree's order (the Hilbert sort
  by itself, for a user who only wants the orders);
* ``search``   -- a batch of queries against a forest that is already built;
* ``batched``  -- many independent sets of uneven size in one segmented forest,
  graph included;
* ``sketch``   -- the second stage: sketches of all points, the sketch-form
  graph and a sketch-form query batch on a forest that is already built;
* ``learned``  -- the per-point budget: the loss and gradients of one training
  batch, the model's predictions for all points, and the budgeted graph.

Points are rows of a Zipf-weighted mixture of anisotropic Gaussians scaled to
unit length (what the repository's benchmark runs on), or unit Gaussian rows
where a case says ``comps`` 0. They are drawn on the GPU from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2508_21682_gb300 as hf

FOREST_SEED = 3


def listed():
    return [
        # the smallest whole job: 20,000 x 16, launches and latency count
        dict(name="graph_tiny", kind="graph", n=20_000, d=16, comps=0, T=8, bits=8, mode=0, slack=-1, w=16, k=10),
        # the plain method at full size, its default budget
        dict(name="graph_plain_3m", kind="graph", n=3_000_000, d=384, comps=1000, T=32, bits=8, mode=0, slack=-1, w=32,
             k=15),
        # the plain method with a wide window on odd sizes: a user who wants
        # recall from few trees, coarse codes, more neighbours
        dict(name="graph_plain_wide", kind="graph", n=100_003, d=100, comps=200, T=8, bits=5, mode=0, slack=-1, w=250,
             k=20),
        # the benchmark's own workload: BF16 Gram form at recall >= 0.8
        dict(name="graph_gram_3m", kind="graph", n=3_000_000, d=384, comps=1000, T=64, bits=8, mode=1, slack=-1, w=1024,
             k=15),
        # a medium set through the BF16 form at a narrow window (one column
        # unit per tile), as an index refreshed often would use
        dict(name="graph_gram_narrow", kind="graph", n=200_001, d=384, comps=200, T=16, bits=8, mode=1, slack=-1, w=48,
             k=10),
        # the orders alone, many short rows: the sort dominates
        dict(name="build_4m", kind="build", n=4_000_037, d=64, comps=1000, T=16, bits=8),
        # the large query batch: 10,000 queries, windows of about 100 points
        dict(name="search_10k", kind="search", n=3_000_000, d=384, comps=1000, T=64, bits=8, nq=10_000, k=30, w=50),
        # a handful of queries, as a service sees them: latency
        dict(name="search_few", kind="search", n=200_000, d=384, comps=200, T=32, bits=8, nq=5, k=10, w=32),
        # independent sets of d = 128 in one forest, the form and window that
        # the autotuner picks for them
        dict(name="batched_128", kind="batched", nsets=23, lo=1000, hi=200_000, d=128, comps=100, T=16, bits=8, mode=1,
             slack=6, w=256, k=10),
        # independent sets of d = 768: the FP8 form with 32 list slots
        dict(name="batched_768_fp8", kind="batched", nsets=16, lo=1000, hi=100_000, d=768, comps=100, T=16, bits=8,
             mode=2, slack=22, w=512, k=10),
        # the sketch stage: graph with the Hamming screen and a query batch
        dict(name="sketch_300k", kind="sketch", n=300_000, d=384, comps=300, T=16, bits=8, sbits=384, w=48, k=15, k2=60,
             nq=2000, ws=128, k2s=300, h=2),
        # the learned budget at work: one training batch, predictions for all
        # points, and the budgeted graph
        dict(name="learned_1m", kind="learned", n=1_000_000, d=384, comps=1000, T=32, bits=8, wmax=512, k=15,
             batch=8192),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["graph", "graph", "graph", "graph", "build", "search", "search", "batched", "sketch", "learned"])
    comps = rng.choice([0, 100, 200, 1000])
    bits = rng.choice([4, 5, 8, 8, 8])
    if kind == "graph":
        mode = rng.choice([0, 0, 0, 1, 1, 2])
        d = rng.choice([16, 33, 64, 100, 128, 129, 200, 256, 384, 384, 384, 500])
        T = _logint(rng, 2, 64)
        w = _logint(rng, 4, 640 if mode == 0 else 1024)
        k = rng.choice([1, 5, 10, 10, 15, 15] + ([20, 30, 50] if mode == 0 else [20, 30]))
        n = _logint(rng, 2000, 3_000_000)
        # no dearer than the largest listed case
        cap = 2.5e11 if mode == 0 else 2e13
        n = int(max(2000, min(n, cap / (float(w + 32) * (d + 32) * T), 6e7 / T)))
        return dict(kind=kind, n=n, d=d, comps=comps, T=T, bits=bits, mode=mode, slack=-1, w=w, k=k)
    if kind == "build":
        d = rng.choice([3, 16, 31, 64, 96, 100, 128, 384])
        T = _logint(rng, 1, 32)
        n = int(min(_logint(rng, 5000, 4_000_037), 6.4e7 / T))
        return dict(kind=kind, n=n, d=d, comps=comps, T=T, bits=bits)
    if kind == "search":
        d = rng.choice([16, 64, 100, 128, 384, 384])
        T = _logint(rng, 2, 64)
        n = int(min(_logint(rng, 5000, 2_000_000), 5e7 / T))
        w = _logint(rng, 8, 128)
        nq = int(max(1, min(_logint(rng, 1, 10_000), 4e10 / (2.0 * w * T * (d + 64)))))
        return dict(kind=kind, n=n, d=d, comps=comps, T=T, bits=bits, nq=nq, k=rng.choice([1, 10, 15, 30, 50]), w=w)
    if kind == "batched":
        d = rng.choice([33, 64, 128, 384, 768])
        mode = 2 if d > 512 else rng.choice([0, 1, 1])
        return dict(kind=kind, nsets=rng.randint(2, 40), lo=rng.choice([50, 1000]), hi=rng.choice([5000, 50_000]), d=d,
                    comps=100, T=rng.choice([4, 8, 16]), bits=8, mode=mode, slack=6 if mode == 1 else (22 if mode == 2 else -1),
                    w=_logint(rng, 16, 64 if mode == 0 else 400), k=10)
    if kind == "sketch":
        return dict(kind=kind, n=_logint(rng, 5000, 300_000), d=rng.choice([100, 128, 384]), comps=max(100, comps),
                    T=_logint(rng, 2, 16), bits=8, sbits=rng.choice([64, 128, 384]), w=_logint(rng, 8, 64), k=15,
                    k2=rng.choice([20, 32, 60]), nq=_logint(rng, 1, 2000), ws=_logint(rng, 16, 128),
                    k2s=rng.choice([60, 300, 500]), h=rng.choice([0, 1, 2]))
    return dict(kind=kind, n=_logint(rng, 20_000, 1_000_000), d=rng.choice([64, 100, 128, 384]), comps=max(100, comps),
                T=_logint(rng, 4, 32), bits=8, wmax=_logint(rng, 32, 512), k=rng.choice([10, 15]),
                batch=rng.choice([1024, 2048, 8192]))


# ---- inputs ---------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _mixture_params(d, comps, seed):
    g = _gen(1_000_003 * seed + 11)
    mu = torch.randn((comps, d), generator=g, device="cuda")
    sg = torch.rand((comps, d), generator=g, device="cuda") * 0.4 + 0.1
    wt = torch.arange(1, comps + 1, device="cuda", dtype=torch.float64) ** -1.1
    return mu, sg, (wt / wt.sum()).cumsum(0).float()


def _rows(n, d, comps, seed, stream, noise=0.0):
    """n x d float32 rows of unit length; the mixture's parameters depend on
    the seed only, the rows on (seed, stream)."""
    g = _gen(1_000_003 * seed + 101 + stream)
    out = torch.empty((n, d), device="cuda")
    par = _mixture_params(d, comps, seed) if comps else None
    for a in range(0, n, 1 << 18):
        b = min(n, a + (1 << 18))
        z = torch.randn((b - a, d), generator=g, device="cuda")
        if par:
            mu, sg, cdf = par
            c = torch.searchsorted(cdf, torch.rand(b - a, generator=g, device="cuda")).clamp_(max=comps - 1)
            z = z * sg[c] + mu[c]
        z /= z.norm(dim=1, keepdim=True)
        if noise:
            z += noise * torch.randn((b - a, d), generator=g, device="cuda")
            z /= z.norm(dim=1, keepdim=True)
        out[a:b] = z
    return out


def _set_offsets(c, seed):
    r = np.random.Generator(np.random.Philox(np.random.SeedSequence([int(seed), 7])))
    sizes = np.rint(np.exp(r.uniform(np.log(c["lo"]), np.log(c["hi"]), size=c["nsets"]))).astype(np.int64)
    # the last set makes the total of every seed the same, so that a case
    # stands for the same amount of work whatever its inputs
    total = int(round((c["hi"] - c["lo"]) / math.log(c["hi"] / c["lo"]) * c["nsets"]))
    sizes = np.maximum(np.floor(sizes * (total / sizes.sum())).astype(np.int64), 2)
    sizes[-1] += max(0, total - int(sizes.sum()))
    return np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)


def _budgets(n, T, wmax, seed):
    """Per-point windows and tree counts as a trained model gives them: most
    points cheap, a tail at the largest budget."""
    g = _gen(1_000_003 * seed + 501)
    lw = 3.0 + (math.log2(wmax) - 3.0) * torch.rand(n, generator=g, device="cuda")
    lt = 1.0 + (math.log2(T) - 1.0) * torch.rand(n, generator=g, device="cuda").sqrt()
    return (torch.exp2(lw).round().clamp_(1, wmax).to(torch.int32), torch.exp2(lt).round().clamp_(1, T).to(torch.int32))


def _targets(c, seed):
    """(log2 w, log2 T) of one training batch."""
    return torch.rand((c["batch"], 2), generator=_gen(1_000_003 * seed + 301), device="cuda") * 5.0 + 2.0


def prepare(case, seed):
    c = dict(case)
    kind = c["kind"]
    st = {"case": c}
    if kind == "batched":
        off = _set_offsets(c, seed)
        st["offsets"] = off
        st["x"] = torch.cat([_rows(int(off[i + 1] - off[i]), c["d"], c["comps"], 64 * seed + i, 0)
                             for i in range(c["nsets"])])
        return st
    st["x"] = _rows(c["n"], c["d"], c["comps"], seed, 0)
    if kind in ("search", "sketch", "learned"):
        st["forest"] = hf.build(st["x"], T=c["T"], bits=c["bits"], seed=FOREST_SEED)
    if kind in ("search", "sketch"):
        st["q"] = _rows(c["nq"], c["d"], c["comps"], seed, 1, noise=0.05)
    if kind == "sketch":
        st["R"] = torch.randn((c["sbits"], c["d"]), generator=_gen(1_000_003 * seed + 401), device="cuda")
        st["forest"].set_option("mode", 3)
        st["forest"].set_option("expand_h", c["h"])
    if kind == "learned":
        st["w_pt"], st["T_pt"] = _budgets(c["n"], c["T"], c["wmax"], seed)
        st["y"] = _targets(c, seed)
        st["mlp"] = hf.Mlp(c["d"], seed=5)
        st["forest"].set_option("mode", 1)
    return st


# ---- one pass -------------------------------------------------------------

def _graph(f, c):
    f.set_option("mode", c["mode"])
    if c["slack"] >= 0:
        f.set_option("tensor_slack", c["slack"])
    return f.knn_graph(c["k"], c["w"])


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "graph":
        with hf.build(state["x"], T=c["T"], bits=c["bits"], seed=FOREST_SEED) as f:
            return _graph(f, c)
    if kind == "build":
        with hf.build(state["x"], T=c["T"], bits=c["bits"], seed=FOREST_SEED) as f:
            out = torch.empty((c["T"], c["n"]), dtype=torch.int32, device="cuda")
            for t in range(c["T"]):
                f.order(t, out=out[t])
            return out
    if kind == "search":
        return state["forest"].search(state["q"], c["k"], c["w"])
    if kind == "batched":
        with hf.build_segmented(state["x"], state["offsets"], T=c["T"], bits=c["bits"], seed=FOREST_SEED) as f:
            return _graph(f, c)
    if kind == "sketch":
        f = state["forest"]
        f.set_sketch(state["R"])
        f.set_option("sketch_k2", c["k2"])
        gi, gd = f.knn_graph(c["k"], c["w"])
        f.set_option("sketch_k2", c["k2s"])
        si, sd = f.search(state["q"], c["k"], c["ws"])
        return gi, gd, si, sd
    loss, grads = state["mlp"].grads(state["x"][:c["batch"]], state["y"])
    pred = state["mlp"].predict(state["x"])
    gi, gd = state["forest"].knn_graph_budget(c["k"], state["w_pt"], state["T_pt"])
    return loss, grads, pred, gi, gd


# ---- what a pass cannot do without -----------------------------------------

def work(case):
    """Inputs read once and outputs written once; operations: the arithmetic of
    the window pairs (each unordered pair of a tree once: 3 d for exact
    differences, 2 d for an inner product), of the scored query candidates and
    of the model."""
    c = case
    kind, d = c["kind"], c["d"]
    if kind == "batched":
        n = int(round((c["hi"] - c["lo"]) / math.log(c["hi"] / c["lo"]) * c["nsets"]))
    else:
        n = c["n"]
    pts = 4.0 * n * d
    if kind in ("graph", "batched"):
        return {"bytes": pts + 8.0 * n * c["k"], "flops": float(n) * c["w"] * c["T"] * d * (3 if c["mode"] == 0 else 2)}
    if kind == "build":
        return {"bytes": pts + 4.0 * n * c["T"], "flops": 0.0}
    if kind == "search":
        # every window row of every tree is read and scored; repeats at most
        # once per point of the matrix
        rows = float(c["nq"]) * 2 * c["w"] * c["T"]
        return {"bytes": 4.0 * d * (min(rows, n) + c["nq"]) + 8.0 * c["nq"] * c["k"], "flops": rows * 3 * d}
    if kind == "sketch":
        words = c["sbits"] / 32
        pairs = float(n) * c["w"] * c["T"]
        cand = n * c["k2"] + c["nq"] * c["k2s"] * (2 * c["h"] + 1)
        return {"bytes": pts + n * words * 4 + 8.0 * n * c["k"] + 8.0 * c["nq"] * c["k"],
                "flops": 2.0 * n * d * c["sbits"] + pairs * words * 3 + cand * 3.0 * d}
    nparam = 256.0 * d + 256 + 65536 + 256 + 512 + 2
    layer = d * 256 + 256 * 256 + 512
    lw, lt = math.log2(c["wmax"]), math.log2(c["T"])
    mw = (c["wmax"] - 8.0) / ((lw - 3.0) * math.log(2)) if lw > 3 else 8.0
    a = (lt - 1.0) * math.log(2)  # mean of 2^(1 + (lt - 1) sqrt(u)), u uniform
    mt = 4.0 * (math.exp(a) * (a - 1.0) + 1.0) / (a * a) if a > 0 else 2.0
    return {"bytes": 2 * pts + 4.0 * c["batch"] * (d + 2) + 4.0 * nparam + 16.0 * n + 8.0 * n * c["k"],
            "flops": 2.0 * n * layer + 6.0 * c["batch"] * layer + float(n) * mw * mt * d * 4.0}


# ---- the same results in 64 bits -------------------------------------------

def _tree_params(seed, tree, d):
    mask = (1 << 64) - 1
    s = (seed + (tree + 1) * 0x9E3779B97F4A7C15) & mask

    def nxt():
        nonlocal s
        s = (s + 0x9E3779B97F4A7C15) & mask
        z = s
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        return z ^ (z >> 31)

    pi = list(range(d))
    for j in range(d - 1, 0, -1):
        m = nxt() % (j + 1)
        pi[j], pi[m] = pi[m], pi[j]
    return pi, [nxt() >> 63 for _ in range(d)]


def _range(x, bits):
    lo, hi = x.amin(0), x.amax(0)
    width = hi - lo
    scale = torch.where(width > 0, (float(1 << bits) / width.double()).float(), torch.zeros_like(width))
    return lo, scale


def _codes(x, lo, scale, bits):
    return ((x - lo) * scale).floor().clamp_(0, (1 << bits) - 1).to(torch.int16)


def _key_words(codes, pi, r, bits):
    """Hilbert keys (rows x d int16 codes) as int32 words of 24 key bits, most
    significant first (Skilling's transposed index)."""
    top = (1 << bits) - 1
    X = [codes[:, p] ^ top if f else codes[:, p].clone() for p, f in zip(pi, r)]
    d = len(X)
    q = 1 << (bits - 1)
    while q > 1:
        low = q - 1
        for i in range(d):
            m = (X[i] & q) != 0
            t = torch.where(m, torch.zeros_like(X[0]), (X[0] ^ X[i]) & low)
            X[0] = torch.where(m, X[0] ^ low, X[0] ^ t)
            if i:
                X[i] = X[i] ^ t
        q >>= 1
    for i in range(1, d):
        X[i] = X[i] ^ X[i - 1]
    t = torch.zeros_like(X[0])
    q = 1 << (bits - 1)
    while q > 1:
        t = torch.where((X[d - 1] & q) != 0, t ^ (q - 1), t)
        q >>= 1
    words, cur, have = [], None, 0
    for lev in range(bits - 1, -1, -1):
        for i in range(d):
            b = ((X[i] ^ t) >> lev) & 1
            cur = b.int() if have == 0 else (cur << 1) | b
            have += 1
            if have == 24:
                words.append(cur)
                have = 0
    if have:
        words.append(cur << (24 - have))
    return words


def _order(words):
    perm = None
    for wd in reversed(words):
        v = wd if perm is None else wd[perm]
        p = torch.sort(v, stable=True).indices
        perm = p if perm is None else perm[p]
    return perm


def _merge(best_d, best_i, d2, cand, k):
    """Top k of the union by (distance, index), repeats dropped."""
    dd, ii = torch.cat([best_d, d2], 1), torch.cat([best_i, cand], 1)
    o = torch.sort(ii, dim=1, stable=True).indices
    dd, ii = dd.gather(1, o), ii.gather(1, o)
    dup = torch.zeros_like(ii, dtype=torch.bool)
    dup[:, 1:] = ii[:, 1:] == ii[:, :-1]
    dd = dd.masked_fill(dup, float("inf"))
    o = torch.sort(dd, dim=1, stable=True).indices[:, :k]
    return dd.gather(1, o), ii.gather(1, o)


def _sq(xa, xb):
    return ((xa - xb) ** 2).sum(-1)


def _exact_graph(case, seed):
    c = case
    n, d, k, w = c["n"], c["d"], c["k"], c["w"]
    x = _rows(n, d, c["comps"], seed, 0)
    codes = _codes(x, *_range(x, c["bits"]), c["bits"])
    xd = x.double()
    bd = torch.full((n, k), float("inf"), dtype=torch.float64, device="cuda")
    bi = torch.full((n, k), n, dtype=torch.int64, device="cuda")
    off = torch.cat([torch.arange(-w, 0), torch.arange(1, w + 1)]).cuda()
    for t in range(c["T"]):
        sig = _order(_key_words(codes, *_tree_params(FOREST_SEED, t, d), c["bits"]))
        step = max(1, int(2e8 / (2 * w * (d + 8))))
        for a in range(0, n, step):
            b = min(n, a + step)
            p = torch.arange(a, b, device="cuda")[:, None] + off
            ok = (p >= 0) & (p < n)
            cand = sig[p.clamp(0, n - 1)]
            me = sig[a:b]
            d2 = _sq(xd[me][:, None, :], xd[cand]).masked_fill(~ok, float("inf"))
            cand = torch.where(ok, cand, torch.full_like(cand, n))
            bd[me], bi[me] = _merge(bd[me], bi[me], d2, cand, k)
    return bd


def _exact_search(case, seed):
    c = case
    n, d, k, w, nq = c["n"], c["d"], c["k"], c["w"], c["nq"]
    x = _rows(n, d, c["comps"], seed, 0)
    q = _rows(nq, d, c["comps"], seed, 1, noise=0.05)
    lo, scale = _range(x, c["bits"])
    allc = torch.cat([_codes(x, lo, scale, c["bits"]), _codes(q, lo, scale, c["bits"])])
    xd, qd = x.double(), q.double()
    bd = torch.full((nq, k), float("inf"), dtype=torch.float64, device="cuda")
    bi = torch.full((nq, k), n, dtype=torch.int64, device="cuda")
    off = torch.arange(-w, w, device="cuda")
    for t in range(c["T"]):
        words = _key_words(allc, *_tree_params(FOREST_SEED, t, d), c["bits"])
        sig = _order([v[:n] for v in words])
        pos = torch.empty(nq, dtype=torch.int64, device="cuda")
        for j in range(nq):  # points with a smaller key than the query's
            less = torch.zeros(n, dtype=torch.bool, device="cuda")
            eq = torch.ones(n, dtype=torch.bool, device="cuda")
            for v in words:
                less |= eq & (v[:n] < v[n + j])
                eq &= v[:n] == v[n + j]
            pos[j] = less.sum()
        p = pos[:, None] + off
        ok = (p >= 0) & (p < n)
        cand = sig[p.clamp(0, n - 1)]
        d2 = _sq(qd[:, None, :], xd[cand]).masked_fill(~ok, float("inf"))
        cand = torch.where(ok, cand, torch.full_like(cand, n))
        bd, bi = _merge(bd, bi, d2, cand, k)
    return bd


def _exact_mlp(x, xb, yb, params, d):
    """(loss, packed gradients of one batch, predictions)."""
    p, o = torch.from_numpy(params).cuda().double().requires_grad_(True), 0

    def take(*shape):
        nonlocal o
        m = math.prod(shape)
        v = p[o:o + m].reshape(shape)
        o += m
        return v

    w1, b1, w2, b2, w3, b3 = take(256, d), take(256), take(256, 256), take(256), take(2, 256), take(2)
    g = torch.nn.functional.gelu

    def net(v):
        return g(g(v.double() @ w1.T + b1) @ w2.T + b2) @ w3.T + b3

    loss = 0.5 * ((net(xb) - yb.double()) ** 2).sum() / xb.shape[0]
    grads, = torch.autograd.grad(loss, p, retain_graph=True)
    with torch.no_grad():
        pred = torch.cat([net(x[a:a + (1 << 16)]) for a in range(0, x.shape[0], 1 << 16)])
    return float(loss), grads.cpu().numpy(), pred


def _mlp_params(d, seed):
    """The model's initial weights (uniform in +-1/sqrt(fan in), splitmix64) in
    the packed order; biases 0."""
    m = 256 * d + 65536 + 512
    i = np.arange(1, m + 1, dtype=np.uint64)
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + i * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    u = ((z >> np.uint64(11)).astype(np.float64) * (1.0 / 9007199254740992.0) * 2.0 - 1.0).astype(np.float32)
    w1 = u[:256 * d] * np.float32(1.0 / np.sqrt(np.float32(d)))
    w2 = u[256 * d:256 * d + 65536] * np.float32(1.0 / 16.0)
    w3 = u[256 * d + 65536:] * np.float32(1.0 / 16.0)
    zero = np.zeros(256, np.float32)
    return np.concatenate([w1, zero, w2, zero, w3, np.zeros(2, np.float32)])


def exact(case, seed):
    """Distances and predictions in 64 bits where that is quick; positions in
    the lists are whole numbers and have no such value."""
    c = case
    # elementwise steps of the key transform (each a few small launches)
    steps = c["d"] * c["bits"] * c["T"]
    if c["kind"] == "graph" and c["mode"] == 0:
        if steps < 100_000 and 2.0 * c["n"] * c["w"] * c["T"] * (c["d"] + 8) < 6e10:
            return None, _exact_graph(c, seed)
    if c["kind"] == "search":
        if steps < 100_000 and float(c["n"]) * steps < 2.5e10 and c["nq"] * c["T"] <= 1000:
            return None, _exact_search(c, seed)
    if c["kind"] == "learned":
        x = _rows(c["n"], c["d"], c["comps"], seed, 0)
        return (*_exact_mlp(x, x[:c["batch"]], _targets(c, seed), _mlp_params(c["d"], 5), c["d"]), None, None)
    return None
