"""Rounds in which whole colour classes have no node: a class whose target
overflowed, then empty classes, then classes that overflow again.  Under every
driver of the rounds, against the oracle's round; whole numbers, every
comparison is for equality."""
import numpy as np
import pytest

import graphgen as gg
import oracle as O

pytestmark = pytest.mark.gpu

S = 64
# classes that are left: neighbours with a gap of one, two and several between
CLASSES = (1, 3, 5, 6, 9, 11, 12, 30, 33, 34, 36, 63)
DRIVERS = {"default": {}, "no_pdl": dict(pdl=0), "serial": dict(concurrent=0),
           "fused": dict(fused_admission=1), "serial_fused": dict(concurrent=0, fused_admission=1)}


@pytest.fixture(params=list(DRIVERS))
def driver(request):
    import paper_1402_3281_gb300 as P
    before = P.get_tuning().to_dict()
    P.set_tuning(**{**before, **DRIVERS[request.param]})
    yield request.param
    P.set_tuning(**before)


def _dev(a):
    import torch
    return None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _class_of(n, rkey):
    """Colour class of every node of a one-graph level."""
    z = np.uint64(rkey) ^ np.arange(n, dtype=np.uint64)
    with np.errstate(over="ignore"):
        z = z + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    z = z ^ (z >> np.uint64(31))
    assert int(z[n - 1]) == O.mix64(rkey ^ (n - 1))
    return (z >> np.uint64(32)) % np.uint64(S)


def _round(g, mode, label, W, bound, rkey):
    import paper_1402_3281_gb300 as P
    import torch
    active = np.isin(_class_of(g.n, rkey), CLASSES).astype(np.uint8)
    ol, oW, om, on = O.lp_round(g, mode, label, W, bound, rkey, S, active_cur=active,
                                want_next=True)
    tl, tW = _dev(label), _dev(W)
    an = torch.zeros(g.n, dtype=torch.uint8, device="cuda")
    moved = P.sclap_lp_round(mode, _dev(g.row_ptr), _dev(g.col), _dev(g.node_w), _dev(g.edge_w),
                             tl, tW, bound, rkey, S, active_cur=_dev(active), active_next=an)
    assert moved == om
    assert np.array_equal(tl.cpu().numpy(), ol)
    assert np.array_equal(tW.cpu().numpy(), oW)
    assert np.array_equal(an.cpu().numpy(), on)
    return om


@pytest.mark.parametrize("leaves", [6000, 20000])     # 20,000: a hub row, never persistent
@pytest.mark.parametrize("weighted", [False, True])
def test_clustering(driver, leaves, weighted):
    """Leaves of a star propose the centre's cluster, which has room for some
    of the first class that is not empty."""
    g = gg.star(leaves)
    if weighted:
        g = gg.random_weights(g, 3, max_node_w=5, max_edge_w=40000)
    W = g.node_w.astype(np.int64)
    label = np.arange(g.n, dtype=np.int32)
    for room in (0, 7, 40, leaves // 20):
        _round(g, O.MODE_CLUSTER, label, W, int(W.max()) + room, 12345 + room)


@pytest.mark.parametrize("over", [0, 2000])
@pytest.mark.parametrize("hub", [False, True])
def test_local_search(driver, over, hub):
    """Three blocks that want to swap many nodes; over > 0 puts block 0 above
    the bound (forced moves, source chain)."""
    g = gg.random_weights(gg.rmat(13, 8, 1), 4)
    if hub:
        n = g.n + 9000
        src = np.repeat(np.arange(g.n), np.diff(g.row_ptr))
        g = gg.random_weights(gg.from_edges(n, np.concatenate([src, np.full(9000, 0)]),
                                            np.concatenate([g.col, np.arange(g.n, n)])), 4)
    rng = np.random.default_rng(over)
    label = rng.integers(0, 3, g.n).astype(np.int32)
    if over:
        label[np.flatnonzero(label != 0)[:over]] = 0
    W = np.bincount(label, weights=g.node_w, minlength=3).astype(np.int64)
    bound = int(W[1:].max()) + (int(g.node_w.sum()) // 50 if over else 30)
    assert bound >= W.max() or over
    assert _round(g, O.MODE_REFINE, label, W, bound, 77) > 0


@pytest.mark.parametrize("graph_rounds", [0, 1])
def test_late_rounds_with_few_active_nodes(driver, graph_rounds):
    import paper_1402_3281_gb300 as P
    g = gg.random_weights(gg.rmat(11, 8, 7), 9)
    kw = dict(sub_rounds=S, cluster_active=1, graph_rounds=graph_rounds)
    dg = [_dev(a) for a in (g.row_ptr, g.col, g.node_w, g.edge_w)]
    ref, rounds = O.cluster(g, 60, seed=4, level=0, cfg=O.config(sub_rounds=S, cluster_active=1))
    got, grounds = P.sclap_cluster(*dg, 60, 4, 0, cfg=P.default_config(**kw))
    assert grounds == rounds and np.array_equal(got.cpu().numpy(), ref)
    k = 5
    Lmax = O.bounds(int(g.node_w.sum()), int(g.node_w.max()), k, 0.03)[0]
    blk = np.random.default_rng(k).integers(0, k, g.n).astype(np.int32)
    ref, rounds = O.refine(g, k, Lmax, blk, seed=5, cfg=O.config(sub_rounds=S))
    got = _dev(blk)
    grounds = P.sclap_refine(*dg, k, Lmax, got, 5,
                             cfg=P.default_config(sub_rounds=S, graph_rounds=graph_rounds))
    assert grounds == rounds and np.array_equal(got.cpu().numpy(), ref)
