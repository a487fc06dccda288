"""Performance cases of the network-embedding library: the calls its users make, through
``paper_2302_07084_gb300.lne`` and ``.search``, over the sizes they make them at.

``listed()`` holds the fixed cases, ``draw(rng)`` gives more of the same ranges,
``prepare(case, seed)`` builds what a program has in hand before the call (a graph on the
GPU, parameters, a context), ``run(state)`` is one pass, ``work(case)`` the bytes and
operations a pass cannot do without, and ``exact(case, seed)`` the pass's result in 64 bits
from plain torch. The restatement of the method here (Philox streams, walks, Eq. 1,
Algorithm 4, the Chebyshev filter, logistic regression) shares no code with the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2302_07084_gb300 import lne, search, synth

BF16 = lne.PREC_BF16_MIXED


# ---------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------

def listed():
    return [
        # one embedding of a very small graph: the library's smoke workload (800 vertices,
        # four blocks, S = 50 per arc, d = 16); launches and host work count
        dict(name="embed_sbm800_d16", kind="embed", graph="sbm", n=800, m=7210, blocks=4, T=10, per_arc=50.0, d=16,
             q=1, k=10),
        # the plain method on the 10,000-vertex, four-block SBM (d = 32, S = 10 T m)
        dict(name="embed_sbm10k_d32", kind="embed", graph="sbm", n=10000, m=119000, blocks=4, T=10, per_arc=50.0,
             d=32, q=1, k=10),
        # the benchmark: BlogCatalog-shaped power-law graph, S = 200 T m = 6.68e8 draws, d = 128
        dict(name="embed_blog_d128", kind="embed", graph="powerlaw", n=10312, m=333983, gamma=2.1, T=10,
             per_arc=1000.0, d=128, q=1, k=10),
        # the sparsifier of a graph whose pairs don't fit a dense table (64-bit keys are
        # sorted), and a product with it: the 10M-vertex run's T = 5, S = 5 T m and exponent
        # at a size that a single call of a pipeline takes
        dict(name="sparsifier_sort_400k", kind="sparsifier", graph="powerlaw", n=400000, m=8000000, gamma=2.2, T=5,
             per_arc=12.5, weighted=False, downsample=False),
        # edge-downsampled draws of a weighted graph (both options that users turn on)
        dict(name="sparsifier_weighted_ds", kind="sparsifier", graph="powerlaw", n=10312, m=333983, gamma=2.1, T=10,
             per_arc=100.0, weighted=True, downsample=True),
        # spectral propagation of a given embedding on the BlogCatalog-shaped graph, FP32
        dict(name="propagate_blog_d128", kind="propagate", graph="powerlaw", n=10312, m=333983, gamma=2.1, d=128,
             k=10, bf16=False),
        # the product of Algorithm 4 with a BF16 operand larger than L2 (c = d + 16 = 144)
        dict(name="spmm_bf16_1m_c144", kind="spmm", n=1000000, m=30000000, gamma=2.2, c=144, bf16=True),
        # orthonormalisation of a tall block of a million rows
        dict(name="cholqr2_1m_c144", kind="cholqr2", n=1000000, c=144),
        # tuning: graphs of the SBM suite, several candidates each, scored by Macro-F1
        dict(name="tune_4x8", kind="tune", graphs=4, n_max=8000, cands=8, d=32),
        # downstream score of one embedding: d = 128, 39 labels, half the vertices for training
        dict(name="macro_f1_blog", kind="macro_f1", n=10312, d=128, labels=39),
        # training the tuning surrogate on 8,192 full runs (100 passes, mini-batches of 256)
        dict(name="surrogate_train_8k", kind="train", rows=8192, epochs=100, batch=256),
        # ranking a pool of 256 candidates with the trained surrogate: the smallest call
        dict(name="surrogate_predict_256", kind="predict", rows=256),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["embed", "embed", "sparsifier", "sparsifier", "propagate", "spmm", "cholqr2", "tune",
                       "macro_f1", "train", "predict"])
    c = dict(kind=kind)
    if kind == "embed":
        if rng.random() < 0.6:
            n = _log(rng, 600, 16000)
            c.update(graph="sbm", n=n, m=int(n * rng.uniform(5.0, 20.0)), blocks=rng.randint(2, 20), T=rng.randint(1, 10),
                     per_arc=round(rng.uniform(20.0, 100.0), 2), d=rng.choice([8, 16, 30, 32, 45, 64]),
                     q=rng.randint(1, 2), k=rng.randint(0, 20))
        else:
            n = _log(rng, 2000, 12000)
            c.update(graph="powerlaw", n=n, m=int(n * rng.uniform(8.0, 30.0)), gamma=round(rng.uniform(2.1, 2.6), 2),
                     T=rng.randint(2, 10), per_arc=round(rng.uniform(20.0, 900.0), 2), d=rng.choice([32, 64, 100, 128]),
                     q=rng.randint(1, 2), k=rng.randint(3, 12))
    elif kind == "sparsifier":
        big = rng.random() < 0.5
        n = _log(rng, 70000, 400000) if big else _log(rng, 1000, 30000)
        m = int(n * rng.uniform(5.0, 20.0))
        c.update(graph="powerlaw", n=n, m=m, gamma=round(rng.uniform(2.1, 2.6), 2), T=rng.randint(1, 10),
                 per_arc=round(min(rng.uniform(2.0, 40.0), 1.0e8 / m), 2), weighted=rng.random() < 0.3,
                 downsample=rng.random() < 0.3)
    elif kind == "propagate":
        n = _log(rng, 1000, 200000)
        bf16 = rng.random() < 0.3
        c.update(graph="powerlaw", n=n, m=int(n * rng.uniform(5.0, 20.0)), gamma=round(rng.uniform(2.1, 2.6), 2),
                 d=rng.choice([16, 32, 64, 128] if bf16 else [16, 32, 50, 64, 128]), k=rng.randint(2, 14), bf16=bf16)
    elif kind == "spmm":
        n = _log(rng, 2000, 1000000)
        bf16 = rng.random() < 0.5
        c.update(n=n, m=int(min(n * rng.uniform(5.0, 60.0), n * n / 8.0, 3.0e7)), gamma=round(rng.uniform(2.1, 2.6), 2),
                 c=4 * rng.randint(2, 36) if bf16 else rng.randint(8, 144), bf16=bf16)
    elif kind == "cholqr2":
        c.update(n=_log(rng, 2000, 1000000), c=rng.randint(8, 144))
    elif kind == "tune":
        c.update(graphs=rng.randint(1, 4), n_max=rng.randint(1500, 8000), cands=rng.randint(2, 8), d=rng.choice([16, 32]))
    elif kind == "macro_f1":
        c.update(n=_log(rng, 1000, 12000), d=rng.randint(16, 128), labels=rng.randint(2, 39))
    elif kind == "train":
        rows, batch = _log(rng, 500, 20000), rng.choice([64, 128, 200, 256, 512])
        passes = min(800000.0, 3000.0 * batch) / rows
        c.update(rows=rows, epochs=max(1, int(rng.uniform(0.1, 1.0) * passes)), batch=batch)
    else:
        c.update(rows=_log(rng, 1, 60000))
    return c


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _sbm_device(n, m, blocks, seed, intra=0.84):
    """About m distinct edges of a block model with equal contiguous blocks, a share
    `intra` of them inside a block, generated on the GPU; (indptr, indices)."""
    g = _gen(seed)
    k = int(m * 1.06) + 16
    u = torch.randint(0, n, (k,), generator=g, device="cuda")
    blk = (u * blocks) // n
    lo = (blk * n + blocks - 1) // blocks
    hi = ((blk + 1) * n + blocks - 1) // blocks
    inside = lo + (torch.rand(k, generator=g, device="cuda", dtype=torch.float64) * (hi - lo)).long()
    anywhere = torch.randint(0, n, (k,), generator=g, device="cuda")
    v = torch.where(torch.rand(k, generator=g, device="cuda") < intra, inside, anywhere)
    ok = u != v
    u, v = u[ok], v[ok]
    keys = torch.unique(torch.cat([u * n + v, v * n + u]))
    rows = keys // n
    indptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.bincount(rows, minlength=n), 0, out=indptr[1:])
    return indptr, (keys % n).to(torch.int32)


def _graph(case, seed):
    if case["graph"] == "sbm":
        return _sbm_device(case["n"], case["m"], case["blocks"], seed)
    return synth.chung_lu_device(case["n"], case["m"], case["gamma"], seed)


def _edge_weights(indptr, indices, seed):
    """Integer weights 1..9, equal on both arcs of an edge (a hash of the pair)."""
    n = indptr.numel() - 1
    src = torch.repeat_interleave(torch.arange(n, device="cuda"), torch.diff(indptr))
    dst = indices.long()
    h = (torch.minimum(src, dst) * 2654435761 + torch.maximum(src, dst) * 40503 + seed * 97) & 0x7FFFFFFF
    h = (h * 1103515245 + 12345) & 0x7FFFFFFF
    return (1 + (h >> 8) % 9).to(torch.int32)


def _device_graph(case, seed):
    indptr, indices = _graph(case, seed)
    g = lne.DeviceGraph.from_tensors(indptr, indices)
    if case.get("weighted"):
        g.weights = _edge_weights(indptr, indices, seed)
    return g


def _params(case, seed, g):
    s = synth.dirichlet_weights(case["T"], seed)
    return lne.Params(T=case["T"], s=list(s), samples=case["per_arc"] * g.nnz, d=case.get("d", 32),
                      q=case.get("q", 1), k=case.get("k", 10), theta=0.5, mu=0.2, seed=seed,
                      downsample_C=lne.default_downsample_C(g.n) if case.get("downsample") else 0.0)


def _embedding(n, d, seed):
    """A U Sigma^{1/2}-like matrix: unit columns of falling scale."""
    x = torch.randn(n, d, generator=_gen(seed), device="cuda")
    x /= x.norm(dim=0)
    return (x * (100.0 ** torch.linspace(1.0, 0.0, d, device="cuda")).sqrt()).contiguous()


def _matrix(case, seed):
    """A sparse symmetric pattern with positive, log-like values."""
    indptr, indices = synth.chung_lu_device(case["n"], case["m"], case["gamma"], seed)
    data = torch.empty(indices.numel(), device="cuda").exponential_(1.0, generator=_gen(seed + 1))
    return dict(n=case["n"], nnz=int(indices.numel()), indptr=indptr, indices=indices, data=data)


def _labelled(case, seed):
    """Embedding rows around label centres; one or two labels a vertex; a half / half split."""
    g, n, d, L = _gen(seed), case["n"], case["d"], case["labels"]
    p = 1.0 / torch.arange(1, L + 1, device="cuda", dtype=torch.float64)
    first = torch.multinomial(p, n, replacement=True, generator=g)
    second = torch.multinomial(p, n, replacement=True, generator=g)
    lab = torch.zeros(n, L, dtype=torch.uint8, device="cuda")
    lab[torch.arange(n, device="cuda"), first] = 1
    two = torch.rand(n, generator=g, device="cuda") < 0.3
    lab[torch.arange(n, device="cuda")[two], second[two]] = 1
    centre = torch.randn(L, d, generator=g, device="cuda")
    x = 0.35 * centre[first] + 0.5 * torch.randn(n, d, generator=g, device="cuda")
    perm = torch.randperm(n, generator=g, device="cuda").to(torch.int32)
    return x.contiguous(), lab, perm[: n // 2].contiguous(), perm[n // 2:].contiguous()


def _candidates(seed, case, m):
    return [lne.Params(T=10, s=list(c["s"]), samples=100.0 * m, d=case["d"], q=1, k=c["k"], theta=c["theta"],
                       mu=c["mu"], seed=seed) for c in synth.tuning_candidates(seed, case["cands"])]


def _tasks(case, seed):
    """Graphs of uneven size, their blocks as labels, a half / half split, candidates."""
    rng = np.random.default_rng(seed)
    tasks, cands = [], []
    for t in range(case["graphs"]):
        n = int(rng.integers(1000, case["n_max"] + 1))
        blocks = int(rng.integers(2, 21))
        m = int(n * rng.uniform(5.0, 20.0))
        indptr, indices = _sbm_device(n, m, blocks, seed * 31 + t, intra=float(rng.uniform(0.35, 0.6)))
        g = _gen(seed * 37 + t)
        lab = torch.zeros(n, blocks, dtype=torch.uint8, device="cuda")
        i = torch.arange(n, device="cuda")
        lab[i, (i * blocks) // n] = 1
        perm = torch.randperm(n, generator=g, device="cuda").to(torch.int32)
        tasks.append((lne.DeviceGraph.from_tensors(indptr, indices), lab, perm[: n // 2].contiguous(),
                      perm[n // 2:].contiguous()))
        cands.append(_candidates(seed * 41 + t, case, indices.numel() // 2))
    return tasks, cands


def _rows(rows, seed):
    """Surrogate inputs (window weights, k, theta, mu, q, 16 graph statistics) and targets."""
    rng = np.random.default_rng(seed)
    s = rng.dirichlet(np.ones(10), rows)
    par = np.stack([rng.integers(3, 21, rows), rng.uniform(0.3, 1.0, rows), rng.uniform(0.0, 0.5, rows),
                    np.ones(rows)], 1)
    graphs = max(1, rows // 32)
    stats = rng.normal(0.0, 1.0, (graphs, 16)) * np.geomspace(0.01, 20.0, 16) + np.linspace(-3.0, 9.0, 16)
    st = stats[np.arange(rows) % graphs]
    x = np.concatenate([s, par, st], 1).astype(np.float32)
    y = 0.2 * s[:, 0] - 0.3 * s[:, 9] + 0.1 * np.sin(par[:, 1] * 5) + 0.02 * par[:, 2] * st[:, 3] \
        + 0.02 * rng.normal(size=rows)
    return x, (y - y.mean()).astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(kind=kind, ctx=lne.Context(0))
    if kind in ("embed", "sparsifier"):
        st["g"] = _device_graph(case, seed)
        st["p"] = _params(case, seed, st["g"])
        if kind == "sparsifier":
            st["X"] = torch.randn(case["n"], 16, generator=_gen(seed + 2), device="cuda")
    elif kind == "propagate":
        st["g"] = _device_graph(case, seed)
        st["p"] = lne.Params(T=1, s=[1.0], samples=1.0, d=case["d"], k=case["k"], theta=0.5, mu=0.2,
                             precision=BF16 if case["bf16"] else lne.PREC_FP32)
        st["X0"] = _embedding(case["n"], case["d"], seed + 7)
    elif kind == "spmm":
        st["M"] = _matrix(case, seed)
        x = torch.randn(case["n"], case["c"], generator=_gen(seed + 2), device="cuda")
        st["X"] = x.to(torch.bfloat16) if case["bf16"] else x
    elif kind == "cholqr2":
        c = case["c"]
        g = _gen(seed)
        mix = torch.linalg.qr(torch.randn(c, c, generator=g, device="cuda"))[0]
        fall = 100.0 ** -torch.linspace(0.0, 1.0, c, device="cuda")
        st["Y"] = (torch.randn(case["n"], c, generator=g, device="cuda") * fall) @ mix
    elif kind == "tune":
        st["tasks"], st["cands"] = _tasks(case, seed)
    elif kind == "macro_f1":
        st["data"] = _labelled(case, seed)
    else:
        x, y = _rows(case["rows"], seed)
        if kind == "train":
            st.update(x=x, y=y, epochs=case["epochs"], batch=case["batch"], seed=seed)
        else:
            rng = np.random.default_rng(seed + 3)
            theta = _network(rng)
            st["ctx"].surrogate_set_params(theta, x.mean(0), np.maximum(x.std(0), 1e-3))
            st["X"] = torch.as_tensor(x).cuda()
    return st


def _network(rng):
    """He-scaled weights of the 30-256-256-1 network, flat."""
    return np.concatenate([rng.normal(0, math.sqrt(2 / 30), 30 * 256), rng.normal(0, 0.05, 256),
                           rng.normal(0, math.sqrt(2 / 256), 65536), rng.normal(0, 0.05, 256),
                           rng.normal(0, math.sqrt(2 / 256), 256), rng.normal(0, 0.05, 1)]).astype(np.float32)


# ---------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------

def run(st):
    ctx, kind = st["ctx"], st["kind"]
    if kind == "embed":
        return ctx.embed(st["g"], st["p"])
    if kind == "sparsifier":   # its entry count varies with the draws: all of it goes into a product
        m = ctx.sparsifier_csr(st["g"], st["p"])
        return dict(indptr=m["indptr"], product=ctx.spmm(m, st["X"]))
    if kind == "propagate":
        return ctx.propagate(st["g"], st["p"], st["X0"])["X"]
    if kind == "spmm":
        return ctx.spmm(st["M"], st["X"])
    if kind == "cholqr2":
        return ctx.cholqr2(st["Y"])
    if kind == "tune":
        return ctx.tune_tasks(st["tasks"], st["cands"])
    if kind == "macro_f1":
        return ctx.macro_f1(*st["data"])
    if kind == "train":
        loss = search.fit_surrogate(ctx, st["x"], st["y"], epochs=st["epochs"], seed=st["seed"], batch=st["batch"])
        return [loss, ctx.surrogate_get_params()]
    return ctx.surrogate_predict(st["X"])


# ---------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind in ("embed", "sparsifier"):
        n, arcs = case["n"], 2.0 * case["m"]
        draws = case["per_arc"] * arcs
        graph = 8.0 * n + arcs * (8.0 if case.get("weighted") else 4.0)
        if kind == "sparsifier":   # a draw's key is written and read once; each entry (col, value) is written
            # and read by the product with 16 columns
            nnz = min(draws, float(n) * n)
            return dict(bytes=graph + 8.0 * draws + 16.0 * nnz + 128.0 * n, flops=32.0 * nnz)
        c, d = case["d"] + 16, case["d"]
        flops = 4.0 * n * c * c * (case["q"] + 2) + 2.0 * arcs * d * (2 * case["k"] + 1) + 8.0 * n * d * d
        return dict(bytes=graph + 8.0 * draws + 4.0 * n * d, flops=flops)
    if kind == "propagate":
        n, d, arcs = case["n"], case["d"], 2.0 * case["m"]
        return dict(bytes=8.0 * n + 4.0 * arcs + 8.0 * n * d, flops=2.0 * arcs * d * (2 * case["k"] - 1) + 8.0 * n * d * d)
    if kind == "spmm":
        n, c, nnz = case["n"], case["c"], 2.0 * case["m"]
        return dict(bytes=8.0 * n + 8.0 * nnz + (6.0 if case["bf16"] else 8.0) * n * c, flops=2.0 * nnz * c)
    if kind == "cholqr2":
        return dict(bytes=8.0 * case["n"] * case["c"], flops=4.0 * case["n"] * case["c"] ** 2)
    if kind == "tune":   # on the mean graph of the range: n, 12.5 edges a vertex, 50 draws an arc
        runs, n = case["graphs"] * case["cands"], (1000 + case["n_max"]) / 2.0
        arcs, d = 25.0 * n, case["d"]
        return dict(bytes=runs * (4.0 * arcs + 8.0 * 50.0 * arcs + 4.0 * n * d),
                    flops=runs * (12.0 * n * (d + 16) ** 2 + 2.0 * arcs * d * 23 + 10.0 * 11 * n / 2 * (d + 1) ** 2))
    if kind == "macro_f1":
        n, d, L = case["n"], case["d"], case["labels"]
        return dict(bytes=4.0 * n * d + n * L + 4.0 * n, flops=10.0 * L * (n / 2.0) * (d + 1) ** 2)
    par = 73985
    if kind == "train":
        return dict(bytes=124.0 * case["rows"] + 12.0 * par, flops=6.0 * par * case["rows"] * case["epochs"])
    return dict(bytes=124.0 * case["rows"] + 2.0 * par, flops=2.0 * par * case["rows"])


# ---------------------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------------------

_M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 on int64 tensors that hold 32-bit words."""
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (((p1 >> 32) & _M32) ^ c1 ^ k0, p1 & _M32, ((p0 >> 32) & _M32) ^ c3 ^ k1, p0 & _M32)
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


def _sources(indptr):
    n = indptr.numel() - 1
    return torch.repeat_interleave(torch.arange(n, device="cuda"), torch.diff(indptr))


def _pair_sums(g, p):
    """(pair keys x n + y, x <= y, sorted; their sample counts or weights in FP64)."""
    n, indptr, dst = g.n, g.indptr, g.indices.long()
    src = _sources(indptr)
    k0, k1 = p.seed & _M32, (p.seed >> 32) & _M32
    arcs = g.nnz
    w = g.weights.long() if g.weights is not None else torch.ones(arcs, dtype=torch.int64, device="cuda")
    deg = torch.zeros(n, dtype=torch.int64, device="cuda").index_add_(0, src, w)
    if g.weights is not None:
        rate = (p.samples * w.double()) / float(deg.sum())
        before = torch.cumsum(w, 0) - w
        upto = torch.cumsum(w, 0) - before[indptr[src]]
        steps = src * (1 << 33) + (upto << 32) // deg[src]
    else:
        rate = torch.full((arcs,), p.samples / arcs, dtype=torch.float64, device="cuda")
    base = torch.floor(rate)
    thr = torch.floor((rate - base) * 4294967296.0).long()
    a = torch.arange(arcs, device="cuda")
    ones = torch.full_like(a, _M32)
    count = base.long() + (_philox(ones, a, torch.zeros_like(a), ones, k0, k1)[0] < thr).long()
    keep_w = None
    if p.downsample_C > 0:
        pe = p.downsample_C * (1.0 / deg[src].double() + 1.0 / deg[dst].double())
        pe = (w.double() * pe if g.weights is not None else pe).clamp(max=1.0)
        coin = torch.floor(pe * 4294967296.0).long()
        keep_w = torch.floor(4294967296.0 / pe + 0.5).long()
    s = np.asarray(p.s, np.float64)
    run_s = np.cumsum(s)
    cut = torch.as_tensor(np.minimum(2.0 ** 32, np.floor(2.0 ** 32 * run_s[:-1] / run_s[-1])).astype(np.int64)).cuda()
    table = torch.zeros(n * n, dtype=torch.int64, device="cuda") if n <= 32768 else None
    parts = []
    step = max(1, int(1.5e7 / max(p.samples / arcs, 1e-9)))
    for a0 in range(0, arcs, step):
        cn = count[a0:a0 + step]
        arc = torch.repeat_interleave(a[a0:a0 + step], cn)
        j = torch.arange(arc.numel(), device="cuda") - torch.repeat_interleave(torch.cumsum(cn, 0) - cn, cn)
        zero = torch.zeros_like(arc)
        block = _philox(j, arc, zero, zero, k0, k1)
        if keep_w is not None:
            on = block[2] < coin[arc]
            arc, j, zero = arc[on], j[on], zero[on]
            block = tuple(b[on] for b in block)
        r = 1 + torch.searchsorted(cut, block[0], right=True)
        sigma = block[1] % r
        u, v = src[arc], dst[arc]
        for t in range(p.T - 1):
            if (3 + t) % 4 == 0:
                block = _philox(j, arc, zero, zero + (3 + t) // 4, k0, k1)
            word, at = block[(3 + t) % 4], torch.where(t < sigma, u, v)
            if g.weights is not None:
                e = torch.searchsorted(steps, at * (1 << 33) + word, right=True).minimum(indptr[at + 1] - 1)
            else:
                e = indptr[at] + word % torch.diff(indptr)[at].clamp(min=1)
            new = torch.where(t < r - 1, dst[e.clamp(max=arcs - 1)], at)
            u, v = torch.where(t < sigma, new, u), torch.where(t < sigma, v, new)
        key = torch.minimum(u, v) * n + torch.maximum(u, v)
        add = keep_w[arc] if keep_w is not None else torch.ones_like(key)
        if table is not None:
            table.index_add_(0, key, add)
        else:
            uk, inv = torch.unique(key, return_inverse=True)
            parts.append((uk, torch.zeros_like(uk).index_add_(0, inv, add)))
    if table is not None:
        keys = torch.nonzero(table).squeeze(1)
        sums = table[keys]
    else:
        keys, inv = torch.unique(torch.cat([q[0] for q in parts]), return_inverse=True)
        sums = torch.zeros_like(keys).index_add_(0, inv, torch.cat([q[1] for q in parts]))
    sums = sums.double()
    return keys, sums * 2.0 ** -32 if keep_w is not None else sums, deg.double()


def _sparsifier64(g, p):
    n = g.n
    keys, K, deg = _pair_sums(g, p)
    x, y = keys // n, keys % n
    vol = float(deg.sum())
    alpha = torch.where(x == y, vol * vol / (p.samples * p.b), vol * vol / (2.0 * p.samples * p.b))
    val = (K * alpha) / (deg[x] * deg[y])
    on = val > 1.0
    x, y, val = x[on], y[on], torch.log(val[on])
    off = x != y
    key = torch.cat([x * n + y, (y * n + x)[off]])
    val = torch.cat([val, val[off]])
    key, order = torch.sort(key)
    indptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.bincount(key // n, minlength=n), 0, out=indptr[1:])
    return indptr, key % n, val[order]


def _csr64(indptr, cols, vals, n):
    return torch.sparse_csr_tensor(indptr, cols.long(), vals.double(), (n, n))


def _left_svd(y):
    u, s, _ = torch.linalg.svd(y, full_matrices=False)
    top = u.abs().argmax(0)
    return u * torch.sign(u[top, torch.arange(u.shape[1], device=u.device)]), s


def _propagate64(g, p, x0):
    if p.k <= 0:
        return x0
    n = g.n
    deg = torch.diff(g.indptr).double()
    a = _csr64(g.indptr, g.indices, torch.ones(g.nnz, device="cuda"), n)
    dinv = torch.where(deg > 0, 1.0 / deg.clamp(min=1.0), torch.zeros_like(deg))[:, None]

    def walk(x):
        return dinv * (a @ x)

    def op(x):
        z = (1.0 - p.mu) * x - walk(x)
        return 0.5 * ((1.0 - p.mu) * z - walk(z)) - x

    def bessel(v):
        return sum((p.theta / 2) ** (2 * t + v) / (math.factorial(t) * math.factorial(t + v)) for t in range(40))

    f, t0, t1 = bessel(0) * x0, x0, None
    for i in range(1, p.k):
        t2 = op(x0) if i == 1 else 2.0 * op(t1) - t0
        t0, t1 = (t0 if i == 1 else t1), t2
        f = f + 2.0 * (-1.0) ** i * bessel(i) * t2
    u, s = _left_svd(walk(x0 - f))
    return u * s.sqrt()


def _embed64(g, p):
    n, c = g.n, p.d + p.oversample
    m = _csr64(*_sparsifier64(g, p), n)
    i = torch.arange(n, device="cuda")[:, None].expand(n, (c + 3) // 4)
    b = torch.arange((c + 3) // 4, device="cuda")[None, :].expand(n, -1)
    zero = torch.zeros_like(i)
    w = [(t.double() + 0.5) / 4294967296.0
         for t in _philox(i, b, zero, zero, (p.seed & _M32) ^ 0x4F4D4547, (p.seed >> 32) & _M32)]
    ra, rb = torch.sqrt(-2.0 * torch.log(w[0])), torch.sqrt(-2.0 * torch.log(w[2]))
    aa, ab = 2.0 * math.pi * w[1], 2.0 * math.pi * w[3]
    y = m @ torch.stack([ra * aa.cos(), ra * aa.sin(), rb * ab.cos(), rb * ab.sin()], 2).reshape(n, -1)[:, :c].contiguous()
    for _ in range(p.q):
        y = m @ torch.linalg.qr(y)[0]
    u, s = _left_svd(y)
    return _propagate64(g, p, (u * s.sqrt())[:, :p.d].contiguous())


def _macro_f1_64(x, lab, train, test):
    x = torch.cat([x.double(), torch.ones(x.shape[0], 1, dtype=torch.float64, device="cuda")], 1)
    xt, y = x[train.long()], lab[train.long()].double() * 2 - 1
    w = torch.zeros(x.shape[1], lab.shape[1], dtype=torch.float64, device="cuda")
    eye = torch.eye(x.shape[1], dtype=torch.float64, device="cuda")
    for _ in range(10):
        sg = torch.sigmoid(y * (xt @ w))
        grad = w + xt.T @ ((sg - 1.0) * y)
        for l in range(lab.shape[1]):
            h = eye + xt.T @ (xt * (sg * (1.0 - sg))[:, l:l + 1])
            w[:, l] -= torch.linalg.solve(h, grad[:, l])
    score, truth = x[test.long()] @ w, lab[test.long()].bool()
    rank = torch.argsort(torch.argsort(-score, dim=1, stable=True), dim=1, stable=True)
    pred = rank < truth.sum(1, keepdim=True)
    tp, fp, fn = (pred & truth).sum(0).double(), (pred & ~truth).sum(0).double(), (~pred & truth).sum(0).double()
    den = 2 * tp + fp + fn
    f1 = torch.where(den > 0, 2 * tp / den.clamp(min=1), torch.zeros_like(den))
    return float(f1.mean()), float(2 * tp.sum() / max(float(den.sum()), 1.0))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("tune", "train"):
        # tune: some tens of whole runs, over the 20 seconds that a value may take here.
        # train: thousands of optimiser steps whose BF16 weight copies round apart
        return None
    st = prepare(case, seed)
    if kind == "embed":
        return _embed64(st["g"], st["p"])
    if kind == "sparsifier":
        indptr, cols, vals = _sparsifier64(st["g"], st["p"])
        return dict(indptr=indptr, product=_csr64(indptr, cols, vals, case["n"]) @ st["X"].double())
    if kind == "propagate":
        return _propagate64(st["g"], st["p"], st["X0"].double())
    if kind == "spmm":
        m = st["M"]
        return _csr64(m["indptr"], m["indices"], m["data"], m["n"]) @ st["X"].double()
    if kind == "cholqr2":
        y = st["Y"].double()
        r = torch.linalg.cholesky(y.T @ y).T.contiguous()
        return torch.linalg.solve_triangular(r, y, upper=True, left=False), r
    if kind == "macro_f1":
        return _macro_f1_64(*st["data"])
    theta, mean, std = st["ctx"].surrogate_get_params()
    t = torch.as_tensor(theta).cuda().to(torch.bfloat16).double()
    x = (st["X"].double() - torch.as_tensor(mean).cuda().double()) / torch.as_tensor(std).cuda().double()
    h = torch.relu(x @ t[:7680].view(30, 256) + t[7680:7936])
    h = torch.relu(h @ t[7936:73472].view(256, 256) + t[73472:73728])
    return h @ t[73728:73984] + t[73984]
