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
