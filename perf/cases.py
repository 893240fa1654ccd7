"""What is timed: the calls that users of this partitioner make.

Each case is one pass through a public entry point on synthetic graphs of the
two families that the repository's benchmark and tests use: R-MAT (skewed
degrees, like web and social graphs; a,b,c,d = 0.57, 0.19, 0.19, 0.05) and 2D
random geometric graphs (meshes; radius 0.55 * sqrt(ln n / n)).  Graphs are
made on the device from the seed alone, so an input costs a second at most.

Every result is a whole number (block ids, cuts, weights).  Only a cut has a
value that plain torch gives without running the method, so `exact` covers
the cut case and is None elsewhere.
"""
import math
import random

import numpy as np
import torch

import paper_1402_3281_gb300 as P

DEV = "cuda"
MAX_NODE_W, MAX_EDGE_W = 4, 8        # the repository's random weights: 1..4 and 1..8


# --------------------------------------------------------------------- cases
def listed():
    return [
        # a caller with one small graph: host and launch latency is all there is
        dict(name="tiny_rmat_2k", kind="partition", family="rmat", n=1 << 10, ef=8, k=2, eps=0.03),
        # the repository's plain single-graph configuration (scale 16, k = 2)
        dict(name="rmat16_k2", kind="partition", family="rmat", n=1 << 16, ef=8, k=2, eps=0.03),
        # a mesh with node and edge weights, a prime node count, an odd block
        # count and a tight balance: finite-element work distribution
        dict(name="rgg_weighted_odd", kind="partition", family="rgg", n=100003, k=13, eps=0.01,
             weighted=True),
        # the throughput configuration: 512 uneven graphs in one call, device arrays
        dict(name="batch512", kind="batch", count=512, sizes=0),
        # host requests through the server, mixed sizes, k and eps
        dict(name="serve48", kind="serve", count=48, sizes=1),
        # the large single-graph configurations (2^22 nodes), one of each family
        dict(name="rmat22_k8", kind="partition", family="rmat", n=1 << 22, ef=16, k=8, eps=0.03),
        dict(name="rgg22_k64", kind="partition", family="rgg", n=1 << 22, k=64, eps=0.03),
        # shaped like a web graph: edge factor 24, k = 16, hubs of 10^5 and more arcs
        dict(name="web24_k16", kind="partition", family="rmat", n=1 << 24, ef=24, k=16, eps=0.03),
        # size-constrained communities without k: clustering and contraction only
        dict(name="communities20", kind="hierarchy", family="rmat", n=1000000, ef=16, bound=4000,
             stop=1000),
        # local search on a partition the caller already has (stripes of a mesh)
        dict(name="refine_stripes", kind="refine", family="rgg", n=1 << 20, k=16, eps=0.03,
             weighted=True),
        # checking a partition: the edge cut of given blocks
        dict(name="cut21_weighted", kind="cut", family="rmat", n=(1 << 21) - 3, ef=16, k=16,
             weighted=True),
        # the quality options: ensembles, three V-cycles, active clustering
        dict(name="quality14", kind="partition", family="rmat", n=1 << 14, ef=8, k=8, eps=0.03,
             quality=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["partition", "partition", "partition", "batch", "serve", "hierarchy",
                       "refine", "cut", "quality"])
    if kind == "batch":
        return dict(kind="batch", count=_log_int(rng, 8, 512), sizes=rng.randrange(1 << 30))
    if kind == "serve":
        return dict(kind="serve", count=_log_int(rng, 4, 48), sizes=rng.randrange(1 << 30))
    c = dict(family=rng.choice(["rmat", "rgg"]))
    k = rng.choice([2, 3, 4, 7, 8, 13, 16, 32, 50, 64])
    weighted = rng.random() < 0.4
    if kind == "quality":
        c.update(kind="partition", n=_log_int(rng, 1 << 11, 1 << 16), k=k, quality=True,
                 eps=rng.choice([0.01, 0.03, 0.05]))
    elif kind == "partition":
        c.update(kind="partition", n=_log_int(rng, 1 << 10, 1 << 22), k=k,
                 eps=rng.choice([0.01, 0.03, 0.05]))
    elif kind == "hierarchy":
        n = _log_int(rng, 1 << 14, 1 << 21)
        c.update(kind="hierarchy", n=n, bound=max(16, n // rng.choice([64, 250, 1000])),
                 stop=rng.choice([500, 1000, 5000]))
    elif kind == "refine":
        c.update(kind="refine", family="rgg", n=_log_int(rng, 1 << 12, 1 << 22), k=k,
                 eps=rng.choice([0.01, 0.03, 0.05]))
    else:
        c.update(kind="cut", n=_log_int(rng, 1 << 12, 1 << 22), k=k)
    if c["family"] == "rmat":
        c["ef"] = rng.choice([8, 16])
    if weighted:
        c["weighted"] = True
    return c


# -------------------------------------------------------------------- graphs
def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed((seed * 1000003 + salt * 7919 + 12345) % (1 << 62))
    return g


def _csr(n, lo, hi, weighted, g):
    """CSR of the undirected edges {lo, hi} (no self-loops; duplicates merged)."""
    key = torch.unique(torch.minimum(lo, hi) * n + torch.maximum(lo, hi))
    w = torch.randint(1, MAX_EDGE_W + 1, key.shape, generator=g, device=DEV,
                      dtype=torch.int32) if weighted else None
    a, b = key // n, key % n
    del key
    both = torch.cat([a * n + b, b * n + a])
    del a, b
    both, order = torch.sort(both)
    if weighted:
        w = torch.cat([w, w])[order]
    del order
    col = (both % n).to(torch.int32)
    src = both // n
    del both
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    row_ptr[1:] = torch.cumsum(torch.bincount(src, minlength=n), 0)
    nw = torch.randint(1, MAX_NODE_W + 1, (n,), generator=g, device=DEV,
                       dtype=torch.int32) if weighted else None
    return dict(row_ptr=row_ptr, col=col, node_w=nw, edge_w=w)


def _rmat(n, ef, weighted, g):
    """R-MAT on the next power of two; n of its ids (chosen at random) kept."""
    scale = max(1, (n - 1).bit_length())
    perm = torch.randperm(1 << scale, generator=g, device=DEV)
    los, his = [], []
    left = ef << scale
    while left > 0:
        m = min(left, 1 << 27)
        left -= m
        s = torch.zeros(m, dtype=torch.int64, device=DEV)
        d = torch.zeros(m, dtype=torch.int64, device=DEV)
        for _ in range(scale):
            r = torch.rand(m, generator=g, device=DEV)
            s = (s << 1) | (r >= 0.76)
            d = (d << 1) | (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
        s, d = perm[s], perm[d]
        keep = (s != d) & (s < n) & (d < n)
        los.append(s[keep])
        his.append(d[keep])
    return _csr(n, torch.cat(los), torch.cat(his), weighted, g)


def _rgg(n, weighted, g):
    """Points in the unit square, cells of the radius' size, pairs of the same
    and of the eight neighbouring cells compared.  Returns the x too."""
    pts = torch.rand(n, 2, generator=g, device=DEV, dtype=torch.float64)
    r = 0.55 * math.sqrt(math.log(n) / n)
    side = max(1, int(1.0 / r))
    cell = (pts * side).long().clamp_(max=side - 1)
    cid, order = torch.sort(cell[:, 0] * side + cell[:, 1])
    sp = pts[order]
    first = torch.searchsorted(cid, torch.arange(side * side + 1, device=DEV))
    cx, cy = cid // side, cid % side
    los, his = [], []
    for dx in (0, 1):                  # a pair is found from its lower cell row
        x = cx + dx
        ok = x < side
        x = x.clamp(max=side - 1)
        a = first[x * side + (cy - 1).clamp(min=0)]
        b = torch.where(ok, first[x * side + (cy + 1).clamp(max=side - 1) + 1], a)
        cnt = b - a
        i = torch.repeat_interleave(torch.arange(n, device=DEV), cnt)
        j = torch.arange(i.numel(), device=DEV) - torch.repeat_interleave(
            torch.cumsum(cnt, 0) - cnt, cnt) + torch.repeat_interleave(a, cnt)
        near = ((sp[i] - sp[j]) ** 2).sum(1) < r * r
        if dx == 0:
            near &= i < j
        los.append(order[i[near]])
        his.append(order[j[near]])
    gr = _csr(n, torch.cat(los), torch.cat(his), weighted, g)
    return gr, pts[:, 0]


def _graph(c, seed, salt=0):
    g = _gen(seed, salt)
    if c["family"] == "rmat":
        return _rmat(c["n"], c["ef"], c.get("weighted", False), g), None
    return _rgg(c["n"], c.get("weighted", False), g)


def _many(c):
    """Sizes, k and eps of the graphs of a batch or of a stream of requests."""
    rng = random.Random(c["sizes"])
    out = []
    for i in range(c["count"]):
        serve = c["kind"] == "serve"
        lo, hi = (12, 17) if serve else (10, 16)
        one = dict(family="rmat", n=1 << rng.randint(lo, hi), ef=8) if i % 2 == 0 else \
            dict(family="rgg", n=_log_int(rng, 4096, 1 << 17) if serve else
                 _log_int(rng, 1000, 65536))
        one["k"] = rng.choice([2, 4, 8, 16, 32, 64] if serve else [2, 4, 8, 16])
        one["eps"] = rng.choice([0.01, 0.03, 0.05]) if serve else 0.03
        out.append(one)
    return out


# ------------------------------------------------------------ prepare and run
def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, seed=seed)
    if kind in ("batch", "serve"):
        gs = []
        for i, one in enumerate(_many(case)):
            gr, _ = _graph(one, seed, i)
            if kind == "serve":
                gr = {q: None if t is None else t.cpu().numpy() for q, t in gr.items()}
            gs.append(dict(gr, k=one["k"], eps=one["eps"], seed=seed + i))
        st["graphs"] = gs
        if kind == "serve":
            st["server"] = P.Server()
        return st
    gr, x = _graph(case, seed)
    st["graph"] = gr
    n = case["n"]
    if case.get("quality"):
        st["cfg"] = P.default_config(ensemble=1, vcycles=3, cluster_active=1)
    if kind == "refine":
        # stripes of equal node counts along x, as a mesh code would start from
        rank = torch.empty(n, dtype=torch.int64, device=DEV)
        rank[torch.argsort(x)] = torch.arange(n, device=DEV)
        st["block"] = (rank * case["k"] // n).to(torch.int32)
        c_v = n if gr["node_w"] is None else int(gr["node_w"].sum())
        st["Lmax"] = math.floor((1.0 + case["eps"]) * -(-c_v // case["k"]))
    if kind == "cut":
        st["block"] = torch.randint(0, case["k"], (n,), generator=_gen(seed, 99), device=DEV,
                                    dtype=torch.int32)
    if gr["col"].numel() > 1 << 26:
        torch.cuda.empty_cache()       # generation needs far more than the graph
    return st


def _args(gr):
    return gr["row_ptr"], gr["col"], gr["node_w"], gr["edge_w"]


def _result(r):
    return dict(block=r.block, cut=r.cut, max_block_weight=r.max_block_weight)


def _results(rs, cat):
    """The results of many graphs, in order, block ids back to back."""
    return dict(block=cat([r.block for r in rs]), cut=np.array([r.cut for r in rs]),
                max_block_weight=np.array([r.max_block_weight for r in rs]))


def run(state):
    case, seed = state["case"], state["seed"]
    kind = case["kind"]
    if kind == "batch":
        return _results(P.sclap_partition_batch(state["graphs"], device=True), torch.cat)
    if kind == "serve":
        srv = state["server"]
        ids = [srv.submit(*_args(g), k=g["k"], eps=g["eps"], seed=g["seed"])
               for g in state["graphs"]]
        return _results([srv.poll(i) for i in ids], np.concatenate)
    gr = state["graph"]
    if kind == "partition":
        return _result(P.sclap_partition_device(*_args(gr), k=case["k"], eps=case["eps"],
                                                seed=seed, cfg=state.get("cfg")))
    if kind == "hierarchy":
        comm, levels, level_n = P.sclap_cluster_hierarchy(*_args(gr), case["bound"],
                                                          case["stop"], seed)
        return dict(comm=comm, levels=levels, level_n=level_n)
    if kind == "refine":
        block = state["block"].clone()
        rounds = P.sclap_refine(*_args(gr), case["k"], state["Lmax"], block, seed)
        return dict(block=block, rounds=rounds)
    return dict(cut=P.sclap_cut(gr["row_ptr"], gr["col"], gr["edge_w"], state["block"]))


# ------------------------------------------------------------- work and exact
def _arcs(c):
    """Expected arcs: 93 % of the sampled R-MAT edges stay after duplicates
    merge (and of those the ones between kept ids); pi * 0.55^2 * ln n
    neighbours in an RGG."""
    if c["family"] == "rmat":
        full = 1 << max(1, (c["n"] - 1).bit_length())
        return 2 * 0.93 * c["ef"] * full * (c["n"] / full) ** 2
    return 0.95 * c["n"] * math.log(c["n"])


def _bytes(c, blocks):
    m, n = _arcs(c), c["n"]
    w = 2 if c.get("weighted") else 1
    return 8 * (n + 1) + 4 * m * w + 4 * n * (w - 1) + 4 * n * blocks


def work(case):
    """The graph read once, the block ids written once (read and written in
    local search, read for a cut).  Integer work: no floating-point operations."""
    if case["kind"] in ("batch", "serve"):
        b = sum(_bytes(one, 1) for one in _many(case))
    else:
        b = _bytes(case, 2 if case["kind"] == "refine" else 1)
    return {"bytes": b, "flops": 0}


def exact(case, seed):
    if case["kind"] != "cut":
        return None
    st = prepare(case, seed)
    gr, blk = st["graph"], st["block"]
    deg = gr["row_ptr"][1:] - gr["row_ptr"][:-1]
    src_blk = torch.repeat_interleave(blk, deg)
    w = torch.ones_like(gr["col"]) if gr["edge_w"] is None else gr["edge_w"]
    cut2 = (w.to(torch.int64) * (src_blk != blk[gr["col"].long()])).sum()
    return dict(cut=int(cut2) // 2)
