"""Every driver of the LP rounds against the oracle: the persistent launch,
launches with and without programmatic edges and side streams, the fused
admission, CUDA-graph rounds, and the launches that a hub row forces.  Nodes
exactly at the edges of every degree bucket, segments of every selection,
several graphs in a level, levels above the persistent rounds' size.  Whole
numbers: every comparison is for equality."""
import functools

import numpy as np
import pytest

import graphgen as gg
import oracle as O
import test_gpu_admission as A
import test_tuning as T

pytestmark = pytest.mark.gpu

# driver: launch setting, rounds as one CUDA graph
DRIVERS = {"default": ({}, 0), "no_pdl": (dict(pdl=0), 0), "serial": (dict(concurrent=0), 0),
           "fused": (dict(fused_admission=1), 0), "graph": ({}, 1),
           "graph_fused": (dict(fused_admission=1), 1)}
LAUNCHED = [d for d in DRIVERS if d != "default"]

# last and first degree of every bucket; 8,192 is the largest row without a hub
EDGES = (4, 5, 8, 9, 16, 17, 32, 33, 128, 129, 512, 513, 2048, 2049, 4096, 4097, 8191, 8192)


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _dg(g):
    return _dev(g.row_ptr), _dev(g.col), _dev(g.node_w), _dev(g.edge_w)


@pytest.fixture
def tuned(request):
    import paper_1402_3281_gb300 as P
    before = P.get_tuning().to_dict()
    setting, graph = DRIVERS[request.param]
    P.set_tuning(**{**before, **setting})
    yield request.param, graph
    P.set_tuning(**before)


def all_drivers(f):
    return pytest.mark.parametrize("tuned", list(DRIVERS), indirect=True)(f)


def all_launched(f):
    return pytest.mark.parametrize("tuned", LAUNCHED, indirect=True)(f)


def launched_by_the_host(f):                          # a single round has no configuration
    names = [d for d in LAUNCHED if not DRIVERS[d][1]]
    return pytest.mark.parametrize("tuned", names, indirect=True)(f)


def _launches(call):
    import paper_1402_3281_gb300 as P
    P.sclap_profile_timeline(True)
    try:
        call()
        return P.sclap_profile_dump()
    finally:
        P.sclap_profile_timeline(False)


@functools.lru_cache(maxsize=None)
def _edge_graph(heavy, hub):
    """One node of each edge degree, its heads drawn from nodes that are not;
    heavy: arc weights whose sums pass 2^32."""
    n = 10000
    edges = EDGES + ((8193, 9000) if hub else ())
    at = 37 * (np.arange(len(edges)) + 1)
    rest = np.setdiff1d(np.arange(n), np.concatenate([at - 1, at, at + 1]))
    rng = np.random.default_rng(4)
    src, dst = [np.arange(n - 1)], [np.arange(1, n)]
    for v, d in zip(at, edges):
        src.append(np.full(d - 2, v))
        dst.append(rng.permutation(rest)[:d - 2])
    g = gg.random_weights(gg.from_edges(n, np.concatenate(src), np.concatenate(dst)), 6,
                          max_edge_w=2 ** 20 if heavy else 8)
    deg = g.degrees()
    for v, d in zip(at, EDGES):
        assert deg[v] == d
    assert (deg.max() > 8192) == hub
    return g


@functools.lru_cache(maxsize=None)
def _reference(heavy, hub, mode, k, S):
    g = _edge_graph(heavy, hub)
    cV = int(g.node_w.sum())
    if mode != "refine":
        U = O.bounds(cV, int(g.node_w.max()), 8, 0.03)[1]
        cfg = O.config(sub_rounds=S, cluster_active=int(mode == "active"))
        return O.cluster(g, U, seed=3, level=1, cfg=cfg) + (U,)
    Lmax = O.bounds(cV, int(g.node_w.max()), k, 0.05)[0]
    blk = np.random.default_rng(k).integers(0, k, g.n).astype(np.int32)
    return O.refine(g, k, Lmax, blk, seed=5, cfg=O.config(sub_rounds=S)) + (Lmax,)


@all_drivers
@pytest.mark.parametrize("hub", [False, True])
@pytest.mark.parametrize("heavy", [False, True])
@pytest.mark.parametrize("mode,k,S", [
    ("cluster", 0, 8), ("cluster", 0, 1), ("active", 0, 64), ("refine", 2, 8),
    ("refine", 257, 64), ("refine", 1025, 3), ("refine", 6000, 8),
])
def test_bucket_edges(tuned, mode, k, S, heavy, hub):
    import paper_1402_3281_gb300 as P
    g = _edge_graph(heavy, hub)
    ref, rounds, bound = _reference(heavy, hub, mode, k, S)
    cfg = P.default_config(sub_rounds=S, cluster_active=int(mode == "active"),
                           graph_rounds=tuned[1])
    if mode != "refine":
        got, grounds = P.sclap_cluster(*_dg(g), bound, 3, 1, cfg=cfg)
    else:
        got = _dev(np.random.default_rng(k).integers(0, k, g.n).astype(np.int32))
        grounds = P.sclap_refine(*_dg(g), k, bound, got, 5, cfg=cfg)
    assert grounds == rounds
    assert np.array_equal(got.cpu().numpy(), ref)


@all_drivers
@pytest.mark.parametrize("hub", [False, True])
def test_the_driver_is_the_one_meant(tuned, hub):
    import paper_1402_3281_gb300 as P
    g = _edge_graph(False, hub)
    d = _launches(lambda: P.sclap_cluster(*_dg(g), 500, 3, 1))
    assert ("k_lp_rounds" in d) == (not hub and tuned[0] in ("default", "graph"))
    assert ("k_resolve" in d or "k_admit" in d) == ("k_lp_rounds" not in d)


@launched_by_the_host
@pytest.mark.parametrize("room", ["none", "one", "some", "all_but_one", "all"])
@pytest.mark.parametrize("leaves", [64, 65, 256, 257, 4096, 4097, 33000])
@pytest.mark.parametrize("weighted", [False, True])
def test_segment_sizes(tuned, leaves, room, weighted):
    A.test_segment_sizes_in_clustering(leaves, room, weighted)


@launched_by_the_host
@pytest.mark.parametrize("over", [0, 1, 2000, 30000])
def test_large_segments(tuned, over):
    A.test_large_segments_in_local_search(over)


@all_launched
@pytest.mark.parametrize("eps", [0.0, 0.03])
def test_batches_and_repair(tuned, eps):
    import paper_1402_3281_gb300 as P
    gs = [gg.rmat(12, 8, 1), gg.rgg2d(3000, 2),
          gg.random_weights(gg.rmat(11, 8, 3), 4, max_node_w=90), gg.path(700), gg.star(900)]
    res = P.sclap_partition_batch([dict(row_ptr=_dev(g.row_ptr), col=_dev(g.col),
                                        node_w=_dev(g.node_w), edge_w=_dev(g.edge_w), k=3 + j,
                                        eps=eps, seed=j) for j, g in enumerate(gs)], device=True,
                                  cfg=P.default_config(graph_rounds=tuned[1]))
    for j, g in enumerate(gs):
        ref = _partition(j, eps)
        assert (res[j].status, res[j].cut) == (ref.status, ref.cut)
        assert np.array_equal(res[j].block.cpu().numpy(), ref.block)


@functools.lru_cache(maxsize=None)
def _partition(j, eps):
    g = [gg.rmat(12, 8, 1), gg.rgg2d(3000, 2),
         gg.random_weights(gg.rmat(11, 8, 3), 4, max_node_w=90), gg.path(700), gg.star(900)][j]
    return O.partition(g, 3 + j, eps, seed=j)


# launch settings that only the launches read, with the persistent rounds off
@pytest.mark.parametrize("si", [i for i, s in enumerate(T.SETTINGS)
                                if {"small_max_deg", "small_ctas_per_sm"} & set(s)])
@pytest.mark.parametrize("off", [dict(pdl=0), dict(fused_admission=1)])
def test_launch_settings(si, off):
    import paper_1402_3281_gb300 as P
    before = P.get_tuning().to_dict()
    gs = T._batch()[:6]                               # (no hub row)
    items = [dict(row_ptr=_dev(g.row_ptr), col=_dev(g.col), node_w=_dev(g.node_w),
                  edge_w=_dev(g.edge_w), k=k, eps=0.03, seed=11 + i) for i, (g, k) in enumerate(gs)]
    try:
        P.set_tuning(**{**before, **T.SETTINGS[si], **off})
        res = P.sclap_partition_batch(items, device=True)
        assert "k_lp_rounds" not in _launches(lambda: P.sclap_partition_batch(items, device=True))
    finally:
        P.set_tuning(**before)
    for i, (g, k) in enumerate(gs):
        ref = _tuning_reference(i)
        assert (res[i].status, res[i].cut) == (ref.status, ref.cut)
        assert np.array_equal(res[i].block.cpu().numpy(), ref.block)


@functools.lru_cache(maxsize=None)
def _tuning_reference(i):
    g, k = T._batch()[i]
    return O.partition(g, k, 0.03, seed=11 + i)


@pytest.mark.parametrize("off", [dict(pdl=0), dict(fused_admission=1)])
def test_thread_launch_split(off):
    """The thread-per-node launch with too few blocks for its three buckets
    (one CTA per SM): the two single-node buckets keep a block each."""
    import paper_1402_3281_gb300 as P
    import torch
    g = T._bucket_mix_graph()
    label = np.arange(g.n, dtype=np.int32)
    W = np.ones(g.n, np.int64)
    ol, oW, om, on = O.lp_round(g, O.MODE_CLUSTER, label, W, 3, 5, 1, want_next=True)
    assert ol[110_000] != 110_000 and ol[110_007] != 110_007
    before = P.get_tuning().to_dict()
    tl, tW = _dev(label), _dev(W)
    an = torch.zeros(g.n, dtype=torch.uint8, device="cuda")
    moved = []
    try:
        P.set_tuning(**{**before, "small_ctas_per_sm": 1, **off})
        d = _launches(lambda: moved.append(P.sclap_lp_round(0, *_dg(g), tl, tW, 3, 5, 1,
                                                            active_next=an)))
    finally:
        P.set_tuning(**before)
    assert "k_propose_small" in d and moved == [om]
    assert np.array_equal(tl.cpu().numpy(), ol)
    assert np.array_equal(tW.cpu().numpy(), oW)
    assert np.array_equal(an.cpu().numpy(), on)


@pytest.mark.parametrize("S,active", [(8, 0), (64, 1)])
def test_above_the_size_of_the_persistent_rounds(S, active):
    """A mesh of 1.25 M nodes and one, launched by default, against the oracle."""
    import paper_1402_3281_gb300 as P
    n, side = 1250001, 1118
    i = np.arange(n)
    right = i[(i % side != side - 1) & (i + 1 < n)]
    down = i[i + side < n]
    g = gg.from_edges(n, np.concatenate([right, down]), np.concatenate([right + 1, down + side]))
    kw = dict(sub_rounds=S, cluster_active=active, lp_rounds_coarse=4)
    ref, rounds = O.cluster(g, 50, seed=9, cfg=O.config(**kw))
    got, grounds = P.sclap_cluster(*_dg(g), 50, 9, cfg=P.default_config(**kw))
    assert grounds == rounds
    assert np.array_equal(got.cpu().numpy(), ref)
