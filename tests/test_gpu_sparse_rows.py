"""Arc and slot streaming over long runs of rows without entries and over
levels with far fewer arcs than rows: equal to a recount and to the oracle,
and no slower for the run than for its rows read once.  Whole numbers: every
comparison is for equality."""
import numpy as np
import pytest

import graphgen as gg
import oracle as O

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _gaps(*parts):
    """A graph of paths (positive lengths) and runs of isolated nodes (negative)."""
    src, n = [], 0
    for p in parts:
        if p > 0:
            src.append(np.arange(n, n + p - 1))
        n += abs(p)
    s = np.concatenate(src)
    return gg.from_edges(n, s, s + 1)


def _spread(n, step):
    s = np.arange(step // 2, n - 1, step)
    return gg.from_edges(n, s, s + 1)


def _ring(n, d):
    """Every node joined to the next d / 2, for odd d every other node to one more."""
    i = np.arange(n)
    src, dst = [np.tile(i, d // 2)], [(i + q) % n for q in range(1, d // 2 + 1)]
    if d % 2:
        src.append(i[::2])
        dst.append((i[::2] + d // 2 + 1) % n)
    return gg.from_edges(n, np.concatenate(src), np.concatenate(dst))


GRAPHS = {f"run_{q}": (lambda q=q: _gaps(700, -q, 900)) for q in (254, 256, 257, 511, 512, 513, 767, 768, 70001)}
# four rows per thread: 1,024 rows a tile
GRAPHS.update({f"quad_{q}": (lambda q=q: _gaps(2, -q, 2, -q, 3, -(q + 1), 2, -4 * q, 5))
               for q in range(1019, 1026)})
# rows of 7, 8 and 9 arcs on average: four rows per thread below 8
GRAPHS.update({f"ring_{d}_{n}": (lambda n=n, d=d: _ring(n, d)) for n in (1023, 1024, 1025, 5000)
               for d in (7, 8, 9)})
GRAPHS.update({
    "run_first": lambda: _gaps(-70001, 3000),
    "run_last": lambda: _gaps(3000, -70001),
    "runs": lambda: _gaps(5, -600, 2, -5000, 4000, -257, 2, -300000, 2, -1, 2, -513, 9),
    "one_edge": lambda: _gaps(-500000, 2, -499999),
    "spread_3": lambda: _spread(300000, 3),
    "spread_257": lambda: _spread(300000, 257),
    "spread_5000": lambda: _spread(2000001, 5000),
})


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_cut_and_contraction(name, weighted):
    import paper_1402_3281_gb300 as P
    g = GRAPHS[name]()
    if weighted:
        g = gg.random_weights(g, 3)
    src = np.repeat(np.arange(g.n), g.degrees())
    dg = (_dev(g.row_ptr), _dev(g.col), _dev(g.node_w) if weighted else None,
          _dev(g.edge_w) if weighted else None)
    blk = np.random.default_rng(g.n).integers(0, 3, g.n).astype(np.int32)
    ref = int(g.edge_w[blk[src] != blk[g.col]].astype(np.int64).sum()) // 2
    assert P.sclap_cut(dg[0], dg[1], dg[3], _dev(blk)) == ref
    # clusters of pairs: runs of coarse nodes without arcs, too
    label = (np.arange(g.n) // 2 * 2).astype(np.int32)
    c = O.contract(g, label)
    cmap, crp, ccol, cnw, cew = P.sclap_contract(*dg, _dev(label))
    assert np.array_equal(cmap.cpu().numpy(), c.cmap)
    assert np.array_equal(cnw.cpu().numpy(), c.node_w)
    crp = crp.cpu().numpy()
    assert np.array_equal(crp, c.row_ptr)
    rows = np.repeat(np.arange(crp.size - 1), np.diff(crp))
    order = lambda col: np.lexsort((col, rows))
    a, b = ccol.cpu().numpy(), c.col
    oa, ob = order(a), order(b)
    assert np.array_equal(a[oa], b[ob])
    assert np.array_equal(cew.cpu().numpy()[oa], c.edge_w[ob])


@pytest.mark.parametrize("at", ["first", "last"])
def test_bad_arc_behind_a_run(at):
    import paper_1402_3281_gb300 as P
    g = _gaps(700, -70001, 900)
    col = g.col.copy()
    col[0 if at == "first" else g.arcs - 1] = g.n
    with pytest.raises(P.SclapError) as e:
        P.sclap_cut(_dev(g.row_ptr), _dev(col), None, _dev(np.zeros(g.n, np.int32)))
    assert e.value.code == P.ECSR


def test_a_run_costs_what_its_rows_cost():
    """Ten million rows without arcs in the middle: staged 256 at a time they
    were tens of milliseconds of one CTA's steps; read once they are 0.1 ms."""
    import time

    import paper_1402_3281_gb300 as P
    import torch
    g = _gaps(1 << 19, -10_000_000, 1 << 19)
    rp, col, blk = _dev(g.row_ptr), _dev(g.col), _dev((np.arange(g.n) % 3).astype(np.int32))
    best = np.inf
    for _ in range(5):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        P.sclap_cut(rp, col, None, blk)
        best = min(best, time.perf_counter() - t0)
    assert best < 0.010
