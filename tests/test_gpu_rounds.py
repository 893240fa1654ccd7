"""The persistent rounds against the launches and the oracle: nodes at the
edges of every degree bucket, many and few labels, one and many colour
classes, sums beyond 32 bits, several graphs in a level, and levels on both
sides of the size at which the launches take over.  Whole numbers: every
comparison is for equality."""
import numpy as np
import pytest

import graphgen as gg
import oracle as O

pytestmark = pytest.mark.gpu

EDGES = (4, 5, 8, 9, 16, 17, 32, 33, 128, 129, 512, 513, 2048, 2049, 8191)


def _dev(a):
    import torch
    return None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _dg(g):
    return _dev(g.row_ptr), _dev(g.col), _dev(g.node_w), _dev(g.edge_w)


def _edge_graph(heavy=False):
    """One node of each edge degree (its heads drawn from the others), on a
    sparse path; heavy: arc weights whose sums pass 2^32."""
    n = 9000
    rng = np.random.default_rng(4)
    src, dst = [np.arange(n - 1)], [np.arange(1, n)]
    for q, d in enumerate(EDGES):
        v = 37 * (q + 1)
        heads = rng.permutation(np.setdiff1d(np.arange(n), [v - 1, v, v + 1]))[:d - 2]
        src.append(np.full(d - 2, v))
        dst.append(heads)
    g = gg.random_weights(gg.from_edges(n, np.concatenate(src), np.concatenate(dst)), 6,
                          max_edge_w=2 ** 20 if heavy else 8)
    return g


@pytest.mark.parametrize("heavy", [False, True])
@pytest.mark.parametrize("mode,k,sub_rounds", [
    ("cluster", 0, 8), ("cluster", 0, 1), ("cluster", 0, 64), ("active", 0, 8),
    ("refine", 2, 8), ("refine", 257, 8), ("refine", 1025, 3), ("refine", 6000, 8),
])
def test_bucket_edges(mode, k, sub_rounds, heavy):
    import paper_1402_3281_gb300 as P
    g = _edge_graph(heavy)
    cV = int(g.node_w.sum())
    kw = dict(sub_rounds=sub_rounds, cluster_active=int(mode == "active"))
    if mode != "refine":
        U = O.bounds(cV, int(g.node_w.max()), 8, 0.03)[1]
        ref, rounds = O.cluster(g, U, seed=3, level=1, cfg=O.config(**kw))
        got, grounds = P.sclap_cluster(*_dg(g), U, 3, 1, cfg=P.default_config(**kw))
    else:
        Lmax = O.bounds(cV, int(g.node_w.max()), k, 0.05)[0]
        blk = np.random.default_rng(k).integers(0, k, g.n).astype(np.int32)
        ref, rounds = O.refine(g, k, Lmax, blk, seed=5, cfg=O.config(**kw))
        got = _dev(blk)
        grounds = P.sclap_refine(*_dg(g), k, Lmax, got, 5, cfg=P.default_config(**kw))
    assert grounds == rounds
    assert np.array_equal(got.cpu().numpy(), ref)


@pytest.mark.parametrize("eps", [0.0, 0.03])
def test_batches_and_repair(eps):
    """Several graphs in a level (done at different rounds), one of them with
    node weights that leave blocks overloaded (forced moves, repair)."""
    import paper_1402_3281_gb300 as P
    gs = [gg.rmat(12, 8, 1), gg.rgg2d(3000, 2), gg.random_weights(gg.rmat(11, 8, 3), 4, max_node_w=90),
          gg.path(700), gg.star(900)]
    res = P.sclap_partition_batch([dict(row_ptr=_dev(g.row_ptr), col=_dev(g.col),
                                        node_w=_dev(g.node_w), edge_w=_dev(g.edge_w), k=3 + j,
                                        eps=eps, seed=j) for j, g in enumerate(gs)], device=True)
    for j, g in enumerate(gs):
        ref = O.partition(g, 3 + j, eps, seed=j)
        assert (res[j].status, res[j].cut) == (ref.status, ref.cut)
        assert np.array_equal(res[j].block.cpu().numpy(), ref.block)


@pytest.mark.parametrize("n", [1249999, 1250001])
def test_both_sides_of_the_size_rule(n):
    """A mesh just below and just above the node limit: the same communities
    as with the launches forced."""
    import paper_1402_3281_gb300 as P
    import torch
    side = 1118
    idx = torch.arange(n, device="cuda")
    right = idx[(idx % side != side - 1) & (idx + 1 < n)]
    down = idx[idx + side < n]
    a = torch.cat([right, down])
    b = torch.cat([right + 1, down + side])
    key, _ = torch.sort(torch.cat([a * n + b, b * n + a]))
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(torch.bincount(key // n, minlength=n), 0)
    col = (key % n).to(torch.int32)
    got, rounds = P.sclap_cluster(rp, col, None, None, 50, 9)
    before = P.get_tuning().to_dict()
    try:
        P.set_tuning(pdl=0)
        ref, rrounds = P.sclap_cluster(rp, col, None, None, 50, 9)
    finally:
        P.set_tuning(**before)
    assert rounds == rrounds
    assert torch.equal(got, ref)
