"""Greedy growing with bitmaps: trial sizes at the edges of a bitmap word, of
the shared-memory bitmaps (32,768 nodes) and of the scans, against the oracle.
Whole numbers: every comparison is for equality."""
import numpy as np
import pytest

import graphgen as gg
import oracle as O

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# trials: 1 and 3 run in wide CTAs; 700 run in narrow ones
@pytest.mark.parametrize("n,k,trials", [
    (2, 2, 3), (31, 3, 3), (32, 2, 700), (33, 4, 700), (64, 2, 3), (1023, 5, 700), (1025, 5, 3),
    (32767, 16, 2), (32768, 16, 2), (32769, 16, 2), (40000, 50, 3),
])
def test_growing_at_bitmap_edges(n, k, trials):
    import paper_1402_3281_gb300 as P
    g = gg.random_weights(gg.rgg2d(n, seed=n) if n > 64 else gg.path(n), 5)
    cV = int(g.node_w.sum())
    avg = -(-cV // k)
    Lmax = O.bounds(cV, int(g.node_w.max()), k, 0.03)[0]
    # no local search: the blocks are the grown ones
    kw = dict(ip_trials=trials, lp_rounds_refine=0)
    ob, ocut, obest = O.initial_partition(g, k, Lmax, avg, seed=7, level=2, cfg=O.config(**kw))
    tb, cut, best = P.sclap_initial_partition(_dev(g.row_ptr), _dev(g.col), _dev(g.node_w),
                                              _dev(g.edge_w), k, Lmax, avg, 7, 2,
                                              cfg=P.default_config(**kw))
    assert (cut, best) == (ocut, obest)
    assert np.array_equal(tb.cpu().numpy(), ob)


# cuts of all trials from one pass over long arc lists: 16 trials fill a word,
# 17 take a second one; more than 256 blocks and short batches take a pass per trial
@pytest.mark.parametrize("scale,factor,trials", [(17, 9, 2), (14, 10, 15), (14, 10, 16), (14, 10, 17),
                                                 (13, 10, 33), (11, 8, 16)])
@pytest.mark.parametrize("k", [2, 255, 256, 257])
def test_best_trial_by_cut(k, scale, factor, trials):
    import paper_1402_3281_gb300 as P
    g = gg.random_weights(gg.rmat(scale, factor, 8), 3, max_edge_w=50)
    cV = int(g.node_w.sum())
    avg = -(-cV // k)
    Lmax = O.bounds(cV, int(g.node_w.max()), k, 0.1)[0]
    kw = dict(ip_trials=trials, lp_rounds_refine=2)
    ob, ocut, obest = O.initial_partition(g, k, Lmax, avg, seed=3, level=1, cfg=O.config(**kw))
    tb, cut, best = P.sclap_initial_partition(_dev(g.row_ptr), _dev(g.col), _dev(g.node_w),
                                              _dev(g.edge_w), k, Lmax, avg, 3, 1,
                                              cfg=P.default_config(**kw))
    assert (cut, best) == (ocut, obest)
    assert np.array_equal(tb.cpu().numpy(), ob)


# two graphs of one batch: each one's arcs and packed words start inside the lists
def test_best_trial_by_cut_batched():
    import paper_1402_3281_gb300 as P
    gs = [gg.random_weights(gg.rmat(14, f, s), s, max_edge_w=50) for f, s in ((9, 4), (7, 5), (8, 6))]
    kw = dict(ip_trials=16, lp_rounds_refine=2, coarse_min_nodes=1 << 15)
    items = [dict(row_ptr=_dev(g.row_ptr), col=_dev(g.col), node_w=_dev(g.node_w),
                  edge_w=_dev(g.edge_w), k=k, eps=0.1, seed=k) for g, k in zip(gs, (3, 5, 16))]
    res = P.sclap_partition_batch(items, cfg=P.default_config(**kw), device=True)
    for g, k, r in zip(gs, (3, 5, 16), res):
        ref = O.partition(g, k, 0.1, seed=k, cfg=O.config(**kw))
        assert (r.status, r.cut) == (ref.status, ref.cut)
        assert np.array_equal(r.block.cpu().numpy(), ref.block)


# copies of a segment: its own weights and offsets, tiles of 1024 arcs, one or many trials
@pytest.mark.parametrize("trials", [1, 2, 5, 16])
def test_copies_of_graphs_that_share_arrays(trials):
    import paper_1402_3281_gb300 as P
    base = gg.rmat(10, 6, 2)
    rp, col = _dev(base.row_ptr), _dev(base.col)
    gs = [gg.random_weights(base, s, max_edge_w=40) for s in (1, 2, 3)]
    kw = dict(ip_trials=trials)
    items = [dict(row_ptr=rp, col=col, node_w=_dev(g.node_w), edge_w=_dev(g.edge_w), k=k,
                  eps=0.1, seed=k) for g, k in zip(gs, (2, 3, 4))]
    items.append(dict(row_ptr=rp, col=col, k=5, eps=0.1, seed=5))
    res = P.sclap_partition_batch(items, cfg=P.default_config(**kw), device=True)
    for g, k, r in zip(gs + [base], (2, 3, 4, 5), res):
        ref = O.partition(g, k, 0.1, seed=k, cfg=O.config(**kw))
        assert (r.status, r.cut) == (ref.status, ref.cut)
        assert np.array_equal(r.block.cpu().numpy(), ref.block)


@pytest.mark.parametrize("n", [1023, 1024, 1025])
@pytest.mark.parametrize("trials", [1, 3, 40])
def test_copies_at_tile_edges(n, trials):
    import paper_1402_3281_gb300 as P
    g = gg.random_weights(gg.rgg2d(n, seed=4), 5)
    k = 3
    cV = int(g.node_w.sum())
    Lmax = O.bounds(cV, int(g.node_w.max()), k, 0.2)[0]
    ob, ocut, obest = O.initial_partition(g, k, Lmax, -(-cV // k), seed=3, level=1,
                                          cfg=O.config(ip_trials=trials))
    tb, cut, best = P.sclap_initial_partition(_dev(g.row_ptr), _dev(g.col), _dev(g.node_w),
                                              _dev(g.edge_w), k, Lmax, -(-cV // k), 3, 1,
                                              cfg=P.default_config(ip_trials=trials))
    assert (cut, best) == (ocut, obest)
    assert np.array_equal(tb.cpu().numpy(), ob)
