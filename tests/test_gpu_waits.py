"""Device-side waits of the default path that run out (their limit lowered by
sclap_debug_inject): the barriers of the persistent rounds and of grouped
growing.  The call reports SCLAP_ETIMEOUT, what it leaves behind is usable,
and the next call equals the oracle.  Nothing here faults or hangs: the waits
are bounded and only their bound is lowered."""
import numpy as np
import pytest

import graphgen as gg
import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture
def P():
    import paper_1402_3281_gb300 as P
    yield P
    P.debug_inject()


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _dg(g):
    return _dev(g.row_ptr), _dev(g.col), _dev(g.node_w), _dev(g.edge_w)


def _times_out(P, call):
    P.debug_inject(wait_limit=1)
    with pytest.raises(P.SclapError) as e:
        call()
    P.debug_inject()
    assert e.value.code == P.ETIMEOUT


def test_clustering(P):
    g = gg.random_weights(gg.rmat(14, 8, 3), 5)
    _times_out(P, lambda: P.sclap_cluster(*_dg(g), 60, 4))
    ref, rounds = O.cluster(g, 60, seed=4)
    got, grounds = P.sclap_cluster(*_dg(g), 60, 4)
    assert grounds == rounds and np.array_equal(got.cpu().numpy(), ref)


def test_local_search(P):
    g = gg.random_weights(gg.rmat(14, 8, 3), 5)
    k = 7
    Lmax = O.bounds(int(g.node_w.sum()), int(g.node_w.max()), k, 0.03)[0]
    blk = np.random.default_rng(1).integers(0, k, g.n).astype(np.int32)
    out = _dev(blk)
    _times_out(P, lambda: P.sclap_refine(*_dg(g), k, Lmax, out, 5))
    left = out.cpu().numpy()
    assert left.min() >= 0 and left.max() < k
    ref, rounds = O.refine(g, k, Lmax, blk, seed=5)
    out = _dev(blk)
    assert P.sclap_refine(*_dg(g), k, Lmax, out, 5) == rounds
    assert np.array_equal(out.cpu().numpy(), ref)


@pytest.mark.parametrize("lp_rounds", [0, 3])
def test_grouped_growing(P, lp_rounds):
    """Two blocks of 2^15 nodes: a group of CTAs grows each trial.  Without
    local search the growing's barriers are the only waits."""
    g = gg.rgg2d(1 << 16, seed=3)
    k = 2
    assert (g.degrees() > 0).sum() // k > 1 << 14
    avg = -(-g.n // k)
    Lmax = O.bounds(g.n, 1, k, 0.03)[0]
    kw = dict(ip_trials=4, lp_rounds_refine=lp_rounds)
    call = lambda: P.sclap_initial_partition(*_dg(g), k, Lmax, avg, 7, 1, cfg=P.default_config(**kw))
    _times_out(P, call)
    ob, ocut, obest = O.initial_partition(g, k, Lmax, avg, seed=7, level=1, cfg=O.config(**kw))
    tb, cut, best = call()
    assert (cut, best) == (ocut, obest)
    assert np.array_equal(tb.cpu().numpy(), ob)


def test_whole_call(P):
    """Every phase of a partition, the rounds after an abandoned one included."""
    g = gg.rmat(16, 8, 1)
    kw = dict(coarse_min_nodes=1 << 15)
    call = lambda: P.sclap_partition_device(*_dg(g), k=2, eps=0.03, seed=3,
                                            cfg=P.default_config(**kw))
    _times_out(P, call)
    ref = O.partition(g, 2, 0.03, seed=3, cfg=O.config(**kw))
    res = call()
    assert (res.status, res.cut) == (ref.status, ref.cut)
    assert np.array_equal(res.block.cpu().numpy(), ref.block)
