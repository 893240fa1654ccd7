"""Arc streaming (csrc/arcs.cuh): cut, validation and block weights at the
sizes where a tile of arcs or of staged rows begins and ends.  Whole numbers:
every comparison is for equality."""
import numpy as np
import pytest

import graphgen as gg

pytestmark = pytest.mark.gpu


def _dev(a, shift=0):
    """CUDA tensor; shift > 0 puts the data off its 16-byte boundary."""
    import torch
    if a is None:
        return None
    a = np.ascontiguousarray(a)
    buf = torch.zeros(a.size + shift, dtype=torch.from_numpy(a[:0]).dtype, device="cuda")
    buf[shift:] = torch.from_numpy(a)
    return buf[shift:]


def _hub_graph(n, hub_deg, gap):
    """Node 0 joined to hub_deg nodes, a run of `gap` isolated nodes, a path
    over the rest."""
    rest = np.arange(1 + gap, n)
    src = np.concatenate([np.zeros(min(hub_deg, rest.size), np.int64), rest[:-1]])
    dst = np.concatenate([rest[:min(hub_deg, rest.size)], rest[1:]])
    return gg.from_edges(n, src, dst)


GRAPHS = {
    "one_arc_pair": lambda: gg.path(2),
    "no_arcs": lambda: gg.from_edges(5, np.zeros(0), np.zeros(0)),
    "tile_minus": lambda: gg.path(1024),          # 2046 arcs: below a tile
    "tile_exact": lambda: gg.path(1025),          # 2048 arcs
    "tile_plus": lambda: gg.path(1026),           # 2050 arcs
    "hub": lambda: _hub_graph(9000, 7001, 0),     # a row of several tiles
    "gap_255": lambda: _hub_graph(5000, 17, 255),
    "gap_256": lambda: _hub_graph(5000, 17, 256),  # a whole tile of empty rows
    "gap_1500": lambda: _hub_graph(5000, 3000, 1500),
    "rmat": lambda: gg.rmat(12, 8, seed=5),
}


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_cut_equals_recount(name, weighted, shift):
    import paper_1402_3281_gb300 as P
    g = GRAPHS[name]()
    g = gg.random_weights(g, 3) if weighted and g.arcs else g
    blk = np.random.default_rng(g.n + shift).integers(0, 3, g.n).astype(np.int32)
    src = np.repeat(np.arange(g.n), g.degrees())
    ref = int(g.edge_w[blk[src] != blk[g.col]].astype(np.int64).sum()) // 2
    col = g.col if g.arcs else np.zeros(1, np.int32)   # a pointer, as the call wants
    got = P.sclap_cut(_dev(g.row_ptr), _dev(col, shift),
                      _dev(g.edge_w, shift) if weighted and g.arcs else None, _dev(blk))
    assert got == ref


@pytest.mark.parametrize("at", ["first", "mid", "last"])
@pytest.mark.parametrize("fault", ["range_high", "range_low", "loop", "weight"])
def test_bad_arc_is_found(fault, at):
    """Every arc of every tile is looked at: a fault in one arc is reported,
    in a batch for its own graph only."""
    import paper_1402_3281_gb300 as P
    g = gg.random_weights(_hub_graph(9000, 7001, 300), 1)
    e = {"first": 0, "mid": 5000, "last": g.arcs - 1}[at]
    src = np.repeat(np.arange(g.n), g.degrees())
    col, ew = g.col.copy(), g.edge_w.copy()
    if fault == "weight":
        ew[e] = 0
    else:
        col[e] = {"range_high": g.n, "range_low": -1, "loop": src[e]}[fault]
    with pytest.raises(P.SclapError) as ei:
        P.sclap_cut(_dev(g.row_ptr), _dev(col), _dev(ew), _dev(np.zeros(g.n, np.int32)))
    assert ei.value.code == P.ECSR
    good = gg.rmat(10, 8, seed=1)
    one = lambda q, c, w: dict(row_ptr=_dev(q.row_ptr), col=_dev(c), edge_w=_dev(w), k=2, seed=4)
    from paper_1402_3281_gb300 import sclap as S
    descs, outs, keep = S._batch_descs([one(good, good.col, good.edge_w), one(g, col, ew),
                                        one(good, good.col, good.edge_w)], True)
    import ctypes as C
    P.load().sclap_partition_batch(3, C.cast(descs, C.c_void_p), None, 1, None)
    assert [d.status for d in descs] == [P.OK, P.ECSR, P.OK]
    alone = P.sclap_partition_device(_dev(good.row_ptr), _dev(good.col), None, _dev(good.edge_w),
                                     k=2, seed=4)
    for j in (0, 2):
        assert descs[j].cut == alone.cut
        assert np.array_equal(outs[j].cpu().numpy(), alone.block.cpu().numpy())


@pytest.mark.parametrize("k", [1, 2, 2048, 2049])
def test_block_weights_on_both_sides_of_the_shared_table(k):
    """Local search from a partition whose blocks sit at the bound: the
    weights decide what may move, and equal the oracle's."""
    import oracle as O
    import paper_1402_3281_gb300 as P
    g = gg.random_weights(gg.rgg2d(6000, seed=2), 2)
    blk = (np.arange(g.n) % k).astype(np.int32)
    Lmax = O.bounds(int(g.node_w.sum()), int(g.node_w.max()), k, 0.03)[0]
    ref, _ = O.refine(g, k, Lmax, blk, seed=3)
    out = _dev(blk)
    P.sclap_refine(_dev(g.row_ptr), _dev(g.col), _dev(g.node_w), _dev(g.edge_w), k, Lmax, out, 3)
    assert np.array_equal(out.cpu().numpy(), ref)
