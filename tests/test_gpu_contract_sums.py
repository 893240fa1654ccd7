"""Contraction on both sides of the total arc weight up to which no coarse
weight can overflow (there the inserts add without a look at the old value):
equal to the oracle, and an edge weight above INT32_MAX is still reported."""
import numpy as np
import pytest

import graphgen as gg
import oracle as O

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _bundle(total):
    """128 edges between two clusters of 64, undirected weights adding to total."""
    i = np.arange(64)
    g = gg.from_edges(128, np.concatenate([i, i]), np.concatenate([i + 64, 64 + (i + 1) % 64]))
    src = np.repeat(np.arange(128), g.degrees())
    lo, hi = np.minimum(src, g.col), np.maximum(src, g.col)
    key = lo.astype(np.int64) * 128 + hi
    w = np.full(128, total // 128, np.int64)
    w[0] += total - w.sum()
    g.edge_w = w[np.searchsorted(np.unique(key), key)].astype(np.int32)
    assert g.edge_w.astype(np.int64).sum() == 2 * total
    return g


# arc weights: twice the total
@pytest.mark.parametrize("total,ok", [((2 ** 31 - 2) // 2, True), (2 ** 30, True),
                                      (2 ** 31 - 1, True), (2 ** 31, False), (2 ** 33, False)])
def test_sums(total, ok):
    import paper_1402_3281_gb300 as P
    g = _bundle(total)
    label = (np.arange(128) // 64 * 64).astype(np.int32)
    call = lambda: P.sclap_contract(_dev(g.row_ptr), _dev(g.col), _dev(g.node_w), _dev(g.edge_w),
                                    _dev(label))
    if not ok:
        with pytest.raises(P.SclapError) as e:
            call()
        assert e.value.code == P.EOVERFLOW
        return
    c = O.contract(g, label)
    cmap, crp, ccol, cnw, cew = (x.cpu().numpy() for x in call())
    assert np.array_equal(crp, c.row_ptr) and np.array_equal(ccol, c.col)
    assert np.array_equal(cew, c.edge_w) and list(cew) == [total, total]
    assert np.array_equal(cnw, c.node_w) and np.array_equal(cmap, c.cmap)
