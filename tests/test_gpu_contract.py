"""Contraction streamed in tiles: regions and rows at tile edges, hubs whose
row and whose coarse region span several tiles, levels on both sides of the
size that waits for its table, unaligned arrays, and the pass ranges.  Whole
numbers, compared for equality with the oracle in a canonical row order."""
import numpy as np
import pytest

import graphgen as gg
import oracle as O

pytestmark = pytest.mark.gpu


def _dev(a, shift=0):
    import torch
    a = np.ascontiguousarray(a)
    buf = torch.zeros(a.size + shift, dtype=torch.from_numpy(a[:0]).dtype, device="cuda")
    buf[shift:] = torch.from_numpy(a)
    return buf[shift:]


def _canon(rp, col, w):
    src = np.repeat(np.arange(rp.size - 1), np.diff(rp))
    o = np.lexsort((col, src))
    return src[o], col[o], w[o]


GRAPHS = {
    "path_2047": lambda: gg.path(1024),
    "path_2050": lambda: gg.path(1026),
    "star_20000": lambda: gg.star(20000),           # one row, and one region, of ten tiles
    "rmat14": lambda: gg.random_weights(gg.rmat(14, 8, 3), 2),
    "isolated": lambda: gg.from_edges(3000, np.arange(2990, 2998), np.arange(2991, 2999)),
}


@pytest.mark.parametrize("table_slots", [0, 1, 700])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("lab", ["own", "pairs", "blocks", "hub_apart", "one"])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_contract_at_tile_edges(name, lab, shift, table_slots):
    import paper_1402_3281_gb300 as P
    g = GRAPHS[name]()
    ids = np.arange(g.n, dtype=np.int32)
    label = {"own": ids, "pairs": ids & ~1, "blocks": ids // 257 * 257,
             "hub_apart": np.where(ids == 0, 0, 1 + (ids - 1) // 3 * 3).astype(np.int32),
             "one": np.zeros(g.n, np.int32)}[lab]
    c = O.contract(g, label)
    before = P.get_tuning().to_dict()
    try:
        P.set_tuning(contract_table_slots=table_slots)
        cmap, crp, ccol, cnw, cew = P.sclap_contract(
            _dev(g.row_ptr), _dev(g.col, shift), _dev(g.node_w), _dev(g.edge_w, shift),
            _dev(label.astype(np.int32)))
    finally:
        P.set_tuning(**before)
    assert np.array_equal(cmap.cpu().numpy(), c.cmap)
    assert np.array_equal(cnw.cpu().numpy(), c.node_w)
    assert np.array_equal(crp.cpu().numpy(), c.row_ptr)
    for x, y in zip(_canon(crp.cpu().numpy(), ccol.cpu().numpy(), cew.cpu().numpy()),
                    _canon(c.row_ptr, c.col, c.edge_w)):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("table_slots", [0, 1 << 20])
@pytest.mark.parametrize("heavy", [False, True])
@pytest.mark.parametrize("arcs", ["4M", "8M"])
def test_contract_of_large_levels(arcs, heavy, table_slots):
    """More than 4 M arcs: table and coarse arrays sized by read-back.  heavy:
    arc weights whose total passes 2^31 (no sums before the table); clusters
    from one node to many tiles."""
    import paper_1402_3281_gb300 as P
    g = gg.rmat(18, 10, 4) if arcs == "4M" else gg.rmat(19, 10, 4)
    assert g.arcs > (4_000_000 if arcs == "4M" else 8_000_000)
    if heavy:
        g = gg.Graph(g.row_ptr, g.col, g.node_w, np.full(g.arcs, 300, np.int32))
    rng = np.random.default_rng(1)
    label = (rng.integers(0, g.n // 40, g.n)).astype(np.int32)
    label[: g.n // 3] = np.arange(g.n // 3)          # singletons
    label[g.n // 3: g.n // 3 + 5000] = 7             # a cluster of many tiles
    c = O.contract(g, label)
    before = P.get_tuning().to_dict()
    try:
        P.set_tuning(contract_table_slots=table_slots)
        cmap, crp, ccol, cnw, cew = P.sclap_contract(
            _dev(g.row_ptr), _dev(g.col), None, _dev(g.edge_w) if heavy else None, _dev(label))
    finally:
        P.set_tuning(**before)
    assert np.array_equal(crp.cpu().numpy(), c.row_ptr)
    for x, y in zip(_canon(crp.cpu().numpy(), ccol.cpu().numpy(), cew.cpu().numpy()),
                    _canon(c.row_ptr, c.col, c.edge_w)):
        assert np.array_equal(x, y)
