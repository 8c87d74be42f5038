"""The work that this framework's users have it do, as cases that can be timed.

Merging proximity graphs (from device or host memory, one at a time or many in a call, with deleted
vertices), building the input graph of a shard, and searching a merged graph (flat and through HNSW
layers). Sizes come from the repository's workloads (synth/gen.py, bench.py) and from its tests;
the data are those workloads' mixtures, drawn on the GPU.
"""
import math

import torch

import paper_2603_21710_gb300 as fg

DEV = "cuda"


# ---------------------------------------------------------------------------- the cases
def listed():
    return [
        # one online lookup in a merged graph of FP32 vectors: what a serving process does per request
        _search("search_one", n=100_000, d=128, data="sift", nq=1),
        # evaluation, or a serving batch: 10,000 queries at once over a quarter of a million vectors
        _search("search_batch", n=250_000, d=128, data="sift", nq=10_000),
        # text embeddings: wide BF16 rows, cosine similarity, a small batch of requests
        _search("search_bf16_cosine", n=100_000, d=768, data="text", dtype="bf16", metric="cos", nq=100, M=24, R=24),
        # the layered search over clustered data, where the flat search starts too far away
        _search("search_layers", n=150_000, d=96, data="deep", metric="ip", nq=1_001, layers=16),
        # two small shards, FP32 rows: a segment merge of a live index, bound by its many short steps
        _merge("merge_small", n=20_000, d=32, data="small", h=2, k=16, R=32, alpha=1.2, M=16, ef=64),
        # the headline workload: a million integer descriptors in four shards
        _merge("merge_sift_1m", n=1_000_000, d=128, data="sift", h=4, k=64, R=32, alpha=1.2, M=32, ef=128),
        # unit-norm float descriptors under inner product, two shards (so a wide search pool)
        _merge("merge_deep_ip", n=300_000, d=96, data="deep", metric="ip", h=2, k=48, R=32, alpha=1.0, M=32, ef=128),
        # high dimension, eight uneven shards, FP8 candidate distances
        _merge("merge_gist_fp8", n=36_000, d=960, data="gist", h=8, split="ragged", k=64, R=48, alpha=1.0, M=32, ef=128,
               join_filter="fp8"),
        # many tenants' merges of uneven size in one call: BF16 embeddings, cosine
        _merge("merge_batch_bf16", n=120_000, d=768, data="text", dtype="bf16", metric="cos", merges=6, h=0, k=32,
               R=24, alpha=1.0, M=24, ef=96),
        # compaction: a quarter of the vertices deleted, three uneven shards of odd sizes
        _merge("merge_deleted", n=99_991, d=128, data="sift", h=3, split="ragged", k=64, R=32, alpha=1.2, M=32, ef=128,
               deleted=0.25),
        # a merge from and to host memory; a dimension and sizes that fit no tile
        _merge("merge_host_odd", n=50_003, d=100, data="deep", h=5, split="ragged", k=30, R=24, alpha=1.1, M=20, ef=80,
               host=True),
        # the input graph of one shard (what every merge needs first)
        dict(name="build_pg", op="build", n=60_000, d=128, data="sift", dtype="f32", metric="l2", M=32, ef=128),
    ]


def _merge(name, n, d, data, h, k, R, alpha, M, ef, dtype="f32", metric="l2", split="even", join_filter="tc", rule="arng",
           deleted=0.0, host=False, merges=1):
    return dict(name=name, op="merge", n=n, d=d, data=data, dtype=dtype, metric=metric, h=h, split=split, k=k, R=R,
                alpha=alpha, M=M, ef=ef, join_filter=join_filter, rule=rule, deleted=deleted, host=host, merges=merges)


def _search(name, n, d, data, nq, dtype="f32", metric="l2", M=32, R=32, beam=64, topk=10, layers=0):
    return dict(name=name, op="search", n=n, d=d, data=data, dtype=dtype, metric=metric, nq=nq, M=M, R=R, beam=beam,
                topk=topk, layers=layers)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search", "search", "search_wide", "layers", "small", "sift", "deep", "gist", "batch", "deleted",
                       "host", "build"])
    if kind == "search":
        data = rng.choice(["sift", "deep"])
        c = _search(None, n=_log(rng, 5_000, 250_000), d=128 if data == "sift" else 4 * rng.randint(8, 32), data=data,
                    nq=_log(rng, 1, 10_000), metric="l2" if data == "sift" else rng.choice(["l2", "ip", "cos"]),
                    R=rng.choice([24, 32, 40]), beam=rng.choice([32, 48, 64, 100, 128]))
    elif kind == "search_wide":
        dt = rng.choice(["f32", "bf16", "bf16"])
        c = _search(None, n=_log(rng, 5_000, 100_000), d=rng.choice([256, 384, 500, 768, 960]), data="text", dtype=dt,
                    metric=rng.choice(["cos", "cos", "ip", "l2"]), nq=_log(rng, 1, 1_000), M=24, R=24,
                    beam=rng.choice([32, 64, 96]))
    elif kind == "layers":
        c = _search(None, n=_log(rng, 10_000, 150_000), d=rng.choice([64, 96, 128]), data="deep", metric="ip",
                    nq=_log(rng, 10, 2_000), layers=rng.choice([8, 16]))
    elif kind == "small":
        c = _merge(None, n=_log(rng, 2_000, 40_000), d=4 * rng.randint(4, 16), data="small", h=rng.randint(2, 4),
                   split=rng.choice(["even", "ragged"]), k=rng.randint(10, 24), R=32, alpha=1.2, M=16, ef=64,
                   rule=rng.choice(["arng", "mrng"]))
    elif kind == "sift":
        c = _merge(None, n=_log(rng, 30_000, 600_000), d=rng.choice([96, 128, 128]), data="sift", h=rng.randint(2, 6),
                   split=rng.choice(["even", "ragged"]), k=rng.choice([32, 48, 64]), R=32, alpha=1.2, M=32, ef=128)
    elif kind == "deep":
        c = _merge(None, n=_log(rng, 20_000, 250_000), d=rng.choice([64, 96, 100, 128]), data="deep",
                   metric=rng.choice(["ip", "l2", "cos"]), h=rng.randint(2, 4), split=rng.choice(["even", "ragged"]),
                   k=rng.randint(32, 64), R=32, alpha=1.0, M=32, ef=128)
    elif kind == "gist":
        c = _merge(None, n=_log(rng, 5_000, 30_000), d=rng.choice([480, 784, 960]), data="gist", h=rng.randint(3, 8),
                   split="ragged", k=rng.choice([40, 64]), R=48, alpha=1.0, M=32, ef=128,
                   join_filter=rng.choice(["fp8", "fp8", "tc"]))
    elif kind == "batch":
        c = _merge(None, n=_log(rng, 20_000, 100_000), d=rng.choice([256, 512, 768]), data="text", dtype="bf16",
                   metric="cos", merges=rng.randint(2, 8), h=0, k=32, R=24, alpha=1.0, M=24, ef=96)
    elif kind == "deleted":
        c = _merge(None, n=_log(rng, 10_000, 200_000), d=128, data="sift", h=rng.randint(2, 5),
                   split=rng.choice(["even", "ragged"]), k=rng.choice([32, 64]), R=32, alpha=1.2, M=32, ef=128,
                   deleted=round(rng.uniform(0.05, 0.4), 3))
    elif kind == "host":
        c = _merge(None, n=_log(rng, 5_000, 100_000), d=4 * rng.randint(10, 32), data=rng.choice(["deep", "small"]),
                   h=rng.randint(2, 6), split="ragged", k=rng.randint(16, 40), R=24, alpha=1.1, M=20, ef=80, host=True)
    else:
        c = dict(name=None, op="build", n=_log(rng, 5_000, 60_000), d=rng.choice([96, 128]),
                 data=rng.choice(["sift", "deep"]), dtype="f32", metric="l2", M=rng.choice([16, 32]),
                 ef=rng.choice([64, 128]))
    del c["name"]
    return c


# ---------------------------------------------------------------------------- inputs
def _points(data, dtype, d, n_centers, counts, seed):
    """[(n, d) points for n in counts] of one seeded mixture."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))

    def normal(*shape):
        return torch.randn(*shape, generator=g, device=DEV)

    def uniform(*shape):
        return torch.rand(*shape, generator=g, device=DEV)

    if data == "sift":        # integer descriptors
        centers, sigma = 255.0 * uniform(n_centers, d), 20.0
    elif data == "small":     # isotropic clusters
        centers, sigma = 20.0 * uniform(n_centers, d) - 10.0, 1.0
    elif data == "deep":      # unit-norm descriptors
        centers, sigma = normal(n_centers, d), 0.5
    elif data == "gist":      # non-negative, high dimension
        centers, sigma = 0.3 * uniform(n_centers, d), 0.05
    elif data == "text":      # unit-norm embeddings, a spread of its own per cluster and dimension
        centers, sigma = normal(n_centers, d), 0.1 + 0.9 * uniform(n_centers, d)
    else:
        raise ValueError(data)
    out = []
    for n in counts:
        c = torch.randint(0, n_centers, (n,), generator=g, device=DEV)
        x = centers[c] + normal(n, d) * (sigma[c] if torch.is_tensor(sigma) else sigma)
        if data == "sift":
            x = x.clamp_(0.0, 255.0).round_()
        elif data == "gist":
            x = x.abs_()
        elif data in ("deep", "text"):
            x = x / x.norm(dim=1, keepdim=True)
        out.append(x.to(torch.bfloat16 if dtype == "bf16" else torch.float32).contiguous())
    return out


def _centers(data, n):
    return 50 if data == "small" else max(10, n // (500 if data in ("deep", "text") else 1000))


def _sizes(n, h, split):
    """Shard sizes: equal, or in the proportion 1 : 2 : ... : h."""
    w = list(range(1, h + 1)) if split == "ragged" else [1] * h
    s = [max(1, n * v // sum(w)) for v in w]
    s[-1] += n - sum(s)
    return s


def _batch_sizes(case):
    """(vertices, shards) of every merge of a call: sizes spread over a factor of eight, 2 to 6 shards."""
    m = case["merges"]
    w = [8.0 ** (i / max(1, m - 1)) for i in range(m)]
    return [(int(case["n"] * v / sum(w)) | 1, 2 + i % 5) for i, v in enumerate(w)]


def _graphs(X, sizes, case):
    adj, entries, o = [], [], 0
    for s in sizes:
        a, e = fg.build_pg(X[o:o + s], M=case["M"], ef=case["ef"], metric=case["metric"])
        adj.append(a)
        entries.append(e)
        o += s
    return adj, entries


def _merge_input(case, n, h, split, seed):
    (X,) = _points(case["data"], case["dtype"], case["d"], _centers(case["data"], n), [n], seed)
    sizes = _sizes(n, h, split)
    adj, entries = _graphs(X, sizes, case)
    return X, sizes, adj, entries


def _merge_args(case):
    return dict(k=case["k"], R=case["R"], alpha=case["alpha"], join_filter=case["join_filter"])


def prepare(case, seed):
    if case["op"] == "search":
        X, Q = _points(case["data"], case["dtype"], case["d"], _centers(case["data"], case["n"]),
                       [case["n"], case["nq"]], seed)
        sizes = _sizes(case["n"], 2, "ragged")
        # a merged graph; the input graphs' pool is narrower than for the merge cases (it is not what is timed)
        adj, entries = _graphs(X, sizes, dict(case, ef=64))
        inp = fg.MergeInput([X[:sizes[0]], X[sizes[0]:]], adj, entries, metric=case["metric"])
        g = fg.merge(inp, k=32, R=case["R"], alpha=1.0, iters=1)
        st = dict(X=X, Q=Q, graph=g["ids"], entry=g["entry"])
        if case["layers"]:
            st["layers"] = fg.build_layers(X, M=case["layers"], ef=64, seed=seed, metric=case["metric"])
    elif case["op"] == "build":
        (X,) = _points(case["data"], case["dtype"], case["d"], _centers(case["data"], case["n"]), [case["n"]], seed)
        st = dict(X=X)
    elif case["merges"] > 1:
        st = dict(inputs=[])
        for i, (n, h) in enumerate(_batch_sizes(case)):
            X, sizes, adj, entries = _merge_input(case, n, h, "even", seed * 64 + i)
            st["inputs"].append(fg.MergeInput.from_flat(X, sizes, torch.cat(adj), entries, metric=case["metric"]))
    else:
        X, sizes, adj, entries = _merge_input(case, case["n"], case["h"], case["split"], seed)
        if case["host"]:
            N = case["n"]
            st = dict(X=X.cpu().pin_memory(), adj=torch.cat(adj).cpu().pin_memory(), sizes=sizes, entries=entries,
                      ids=torch.empty((N, case["R"]), dtype=torch.int32).pin_memory(),
                      deg=torch.empty((N,), dtype=torch.int32).pin_memory())
        else:
            valid = None
            if case["deleted"]:
                g = torch.Generator(device=DEV).manual_seed(int(seed) + 7)
                valid = torch.ones(case["n"], dtype=torch.bool, device=DEV)
                valid[torch.randperm(case["n"], generator=g, device=DEV)[:int(case["deleted"] * case["n"])]] = False
            st = dict(inp=fg.MergeInput.from_flat(X, sizes, torch.cat(adj), entries, metric=case["metric"], valid=valid))
    st["case"] = case
    return st


# ---------------------------------------------------------------------------- one pass
def _graph(out):
    return {"ids": out["ids"], "dist": out["dist"], "deg": out["deg"], "entry": out["entry"]}


def run(st):
    c = st["case"]
    if c["op"] == "search":
        if c["layers"]:
            ly = st["layers"]
            ids, dist, _ = fg.search_hnsw(st["X"], st["graph"], ly["layers"], ly["entry"], st["Q"], topk=c["topk"],
                                          beam=c["beam"], metric=c["metric"])
        else:
            ids, dist = fg.search(st["X"], st["graph"], st["entry"], st["Q"], topk=c["topk"], beam=c["beam"],
                                  metric=c["metric"])
        return {"ids": ids, "dist": dist}
    if c["op"] == "build":
        adj, entry = fg.build_pg(st["X"], M=c["M"], ef=c["ef"], metric=c["metric"])
        return {"adj": adj, "entry": entry}
    if c["merges"] > 1:
        return [_graph(o) for o in fg.merge_batch(st["inputs"], **_merge_args(c))]
    if c["host"]:
        out = fg.merge_host(st["X"], st["adj"], st["sizes"], st["entries"], metric=c["metric"], out_ids=st["ids"],
                            out_deg=st["deg"], **_merge_args(c))
        return {"ids": out["ids"], "deg": out["deg"], "entry": out["entry"]}
    return _graph(fg.merge(st["inp"], rule=c["rule"], **_merge_args(c)))


# ---------------------------------------------------------------------------- what a pass cannot do without
def work(case):
    """Inputs read once, outputs written once, and the distances of the searches and of the graph step.

    A search with a pool of L over a graph of degree M expands at least L vertices; about half of
    their neighbours have been met before. The refinement and the selection are counted by the
    distances of a vertex to its k list entries' lists once per pass, of which half are new."""
    d, row = case["d"], case["d"] * (2 if case["dtype"] == "bf16" else 4)
    per = 3 * d if case["metric"] == "l2" else 2 * d
    n = case["n"]
    if case["op"] == "search":
        evals = min(n, case["beam"] * case["R"] // 2)
        rows = min(n, case["nq"] * evals)
        hops = min(n, case["nq"] * case["beam"])
        return {"bytes": rows * row + hops * case["R"] * 4 + case["nq"] * (row + 8 * case["topk"]),
                "flops": case["nq"] * evals * per}
    if case["op"] == "build":
        return {"bytes": n * (row + case["M"] * 4), "flops": n * min(n, case["ef"] * case["M"] // 2) * per}
    h = case["h"] or 4
    L = -(-case["k"] // (h - 1))
    evals = (h - 1) * L * case["M"] // 2 + case["k"] * case["k"] // 2
    return {"bytes": n * (row + case["M"] * 4 + 8 * case["R"] + 4), "flops": n * evals * per}


# ---------------------------------------------------------------------------- the same in 64 bits
def _pool_search(X, adj, start, Q, metric, L):
    """Best-first search of every query at once: pools of L (distance, id), ascending, in 64 bits."""
    nq, inf = Q.shape[0], float("inf")

    def dist(i):   # [nq, m] distances to the rows i
        x = X[i.clamp_min(0)]
        if metric == "l2":
            return (x - Q[:, None, :]).square().sum(-1)
        return 1.0 - torch.einsum("qmd,qd->qm", x, Q)

    pi = torch.full((nq, L), -1, dtype=torch.int64, device=DEV)
    pd = torch.full((nq, L), inf, dtype=torch.float64, device=DEV)
    pe = torch.zeros((nq, L), dtype=torch.bool, device=DEV)
    pi[:, 0] = start
    pd[:, :1] = dist(pi[:, :1])
    rows = torch.arange(nq, device=DEV)
    while True:
        open_ = (pi >= 0) & ~pe
        act = open_.any(1)
        if not bool(act.any()):
            return pi, pd
        f = open_.int().argmax(1)
        pe[rows, f] |= act
        nb = adj[pi[rows, f].clamp_min(0)].long()
        ok = (nb >= 0) & act[:, None] & ~(nb[:, :, None] == pi[:, None, :]).any(-1)
        nd = torch.where(ok, dist(nb), inf)
        ai = torch.cat([pi, torch.where(ok, nb, -1)], 1)
        ad, ae = torch.cat([pd, nd], 1), torch.cat([pe, torch.zeros_like(ok)], 1)
        o = torch.sort(ai, dim=1, stable=True).indices
        o = o.gather(1, torch.sort(ad.gather(1, o), dim=1, stable=True).indices)[:, :L]
        pi, pd, pe = ai.gather(1, o), ad.gather(1, o), ae.gather(1, o)
        pi = torch.where(torch.isinf(pd), -1, pi)


def exact(case, seed):
    """The searches in 64 bits. The merges and the graph builder have no quick 64-bit form; what they
    return are ids, and distances that are held to the start's."""
    if case["op"] != "search":
        return None
    st = prepare(case, seed)
    X, Q, metric = st["X"].double(), st["Q"].double(), case["metric"]
    if metric == "cos":
        X, Q = X / X.norm(dim=1, keepdim=True), Q / Q.norm(dim=1, keepdim=True)
    start = torch.full((case["nq"],), st["entry"], dtype=torch.int64, device=DEV)
    if case["layers"]:
        start.fill_(st["layers"]["entry"])
        for ly in reversed(st["layers"]["layers"]):
            mem = ly["members"].long()
            at = torch.searchsorted(mem, start)
            start = mem[_pool_search(X[mem], ly["adj"], at, Q, metric, 8)[0][:, 0]]
    i, v = _pool_search(X, st["graph"], start, Q, metric, case["beam"])
    return {"ids": None, "dist": v[:, :case["topk"]]}
