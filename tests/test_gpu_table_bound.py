"""The contraction table of a small level is taken at its largest size without
asking for it: two slots per arc, which rows of one and of two coarse arcs
need to the last slot.  Equal to the oracle, and taken that way as soon as the
slots allowed per pass reach that bound."""
import numpy as np
import pytest

import graphgen as gg
import oracle as O

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("slots", [0, -1])           # exactly the bound, one below it
@pytest.mark.parametrize("rows", [1, 2, 3])
def test_largest_table(rows, slots):
    import paper_1402_3281_gb300 as P
    n = 6000
    i = np.arange(n)
    if rows == 1:                                     # a perfect matching
        g = gg.from_edges(n, i[::2], i[1::2])
    elif rows == 2:                                   # a cycle
        g = gg.from_edges(n, i, (i + 1) % n)
    else:                                             # a cycle with its diameters
        g = gg.from_edges(n, np.concatenate([i, i[:n // 2]]),
                          np.concatenate([(i + 1) % n, i[:n // 2] + n // 2]))
    assert (g.degrees() == rows).all()
    label = i.astype(np.int32)                        # no cluster of two: nothing merges
    c = O.contract(g, label)
    before = P.get_tuning().to_dict()
    try:
        P.set_tuning(**{**before, "contract_table_slots": 2 * g.arcs + slots})
        P.sclap_profile_timeline(True)
        cmap, crp, ccol, cnw, cew = P.sclap_contract(_dev(g.row_ptr), _dev(g.col), _dev(g.node_w),
                                                     _dev(g.edge_w), _dev(label))
        launched = P.sclap_profile_dump()
    finally:
        P.sclap_profile_timeline(False)
        P.set_tuning(**before)
    assert ("k_clear_table" in launched) == (slots == 0)
    crp = crp.cpu().numpy()
    assert np.array_equal(cmap.cpu().numpy(), c.cmap) and np.array_equal(crp, c.row_ptr)
    src = np.repeat(np.arange(n), np.diff(crp))
    o, p = np.lexsort((ccol.cpu().numpy(), src)), np.lexsort((c.col, src))
    assert np.array_equal(ccol.cpu().numpy()[o], c.col[p])
    assert np.array_equal(cew.cpu().numpy()[o], c.edge_w[p])
