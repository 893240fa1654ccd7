"""Admission of one colour class: segments at the edges of the warp (64
entries), CTA (4,096) and cluster selections, with the boundary at the first,
an inner and the last entry.  Against the oracle's round; whole numbers, every
comparison is for equality."""
import numpy as np
import pytest

import graphgen as gg
import oracle as O

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _round(g, mode, label, W, bound, rkey):
    """One round with a single colour class, on the GPU and by the oracle."""
    import paper_1402_3281_gb300 as P
    import torch
    ol, oW, om, on = O.lp_round(g, mode, label, W, bound, rkey, 1, want_next=True)
    tl, tW = _dev(label), _dev(W)
    an = torch.zeros(g.n, dtype=torch.uint8, device="cuda")
    moved = P.sclap_lp_round(mode, _dev(g.row_ptr), _dev(g.col), _dev(g.node_w), _dev(g.edge_w),
                             tl, tW, bound, rkey, 1, active_next=an)
    assert moved == om
    assert np.array_equal(tl.cpu().numpy(), ol)
    assert np.array_equal(tW.cpu().numpy(), oW)
    assert np.array_equal(an.cpu().numpy(), on)
    return om


@pytest.mark.parametrize("room", ["none", "one", "some", "all_but_one", "all"])
@pytest.mark.parametrize("leaves", [63, 64, 65, 4095, 4096, 4097, 33000])
@pytest.mark.parametrize("weighted", [False, True])
def test_segment_sizes_in_clustering(leaves, room, weighted):
    """Every leaf of a star proposes the centre's cluster: one segment.  With
    weights the gains differ (several key digits), without them only the
    priority hash orders the entries."""
    g = gg.star(leaves)
    if weighted:
        g = gg.random_weights(g, 3, max_node_w=5, max_edge_w=40000)
    label = np.arange(g.n, dtype=np.int32)
    W = g.node_w.astype(np.int64)
    # the centre may not move: it is heavier than any leaf cluster's room
    total = int(W[1:].sum())
    extra = {"none": 0, "one": int(W.max()), "some": total // 3, "all_but_one": total - 1,
             "all": total}[room]
    bound = int(W[0]) + extra
    _round(g, O.MODE_CLUSTER, label, W, bound, 12345 + leaves)


@pytest.mark.parametrize("over", [0, 1, 2000, 30000])
def test_large_segments_in_local_search(over):
    """Two blocks that want to swap many nodes: target segments of thousands;
    over > 0 puts block 0 above the bound (forced moves, source chain)."""
    g = gg.random_weights(gg.rmat(16, 8, 1), 4)
    rng = np.random.default_rng(over)
    label = rng.integers(0, 3, g.n).astype(np.int32)
    W = np.bincount(label, weights=g.node_w, minlength=3).astype(np.int64)
    if over:
        mv = np.flatnonzero(label != 0)[:over]
        label[mv] = 0
        W = np.bincount(label, weights=g.node_w, minlength=3).astype(np.int64)
        bound = int(W[1:].max()) + int(g.node_w.sum()) // 50
    else:
        bound = int(W.max()) + 1000
    assert _round(g, O.MODE_REFINE, label, W, bound, 77) > 0
