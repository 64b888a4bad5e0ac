"""The kernels of a round at the sizes where their tiling can go wrong, against the oracle (exact)."""
import numpy as np
import pytest

import oracle
import synth
from parity_util import compare_state

pytestmark = pytest.mark.gpu


LAUNCHES = 32   # debug bit: the launches of large instances whatever the size


def _check(hg, rounds=4, subrounds=4, eps=None, **kw):
    """Both ways a small instance can run: as one cluster, and by the launches of large ones."""
    from paper_2010_10272_gb300 import HGP
    if eps is not None:
        hg.eps = eps
    o = oracle.Oracle.from_hypergraph(hg, subrounds=subrounds, seed=9, **kw)
    want, _ = o.refine(rounds)
    for debug in (0, LAUNCHES):
        h = HGP.from_hypergraph(hg, subrounds=subrounds, seed=9, debug=debug, **kw)
        got = np.concatenate([h.refine(1), h.refine(rounds - 1)])
        assert np.array_equal(got[:, :5], want[:, :5])
        compare_state(h, o)
        h.close()


@pytest.mark.parametrize("n", [2047, 2048, 2049, 4096, 6145, 33_000])
@pytest.mark.parametrize("weighted", [False, True])
def test_ties_at_the_threshold_gain(n, weighted):
    """Small nets give few distinct gains, so a saturated block's budget ends inside a long run of
    equal gains: the last approved id falls anywhere in a tile of 2048 vertices."""
    hg = synth.random_small(n, n, n, 5, max_size=3, weighted=weighted, f=0.9)
    _check(hg, eps=0.004)
    _check(hg, eps=0.004, subrounds=1)


@pytest.mark.parametrize("k", [2, 32, 33, 64])
@pytest.mark.parametrize("m,scale", [(2_000, 0), (8_000, 0), (8_000, 1), (8_000, 6), (30_000, 0), (2_000, 1_000_000)])
@pytest.mark.parametrize("balance", [False, True])
def test_degrees_and_net_weights(k, m, scale, balance):
    """300 vertices of about 23, 93 and 350 nets: below, around and above the degree (96) from which a
    warp walks a vertex's nets together; net weights (scale > 0) put W(u) around and above 2047, the
    last value the bit planes hold."""
    hg = synth.random_small(k, 300, m, k, max_size=6, weighted=True, f=0.6)
    hg.net_w = (hg.net_w * scale).astype(np.int32) if scale else None
    hg.vertex_w = (hg.vertex_w * 3 - 2).astype(np.int32)      # 1..13: beside the weights with a mask of their own
    _check(hg, eps=0.2, balance_moves=balance)


@pytest.mark.parametrize("S", [1, 2, 3, 7, 64])
def test_tiles_and_segments(S):
    """Sub-round lists of whole, partial and single-vertex tiles (2048 vertices) cut into segments of
    32, alone and as members of one batch, and rebalancing from an overloaded start."""
    from paper_2010_10272_gb300 import HGP, Batch
    hgs = [synth.random_small(7 * n + S, n, n + 3, k, max_size=5, weighted=n % 2 == 0, f=0.7)
           for n, k in ((4, 2), (31, 3), (2048, 40), (2049, 5), (5000, 16), (5000, 64))]
    for hg in hgs:
        _check(hg, rounds=3, subrounds=S)
    subs = [S, S, S, 2, S, S]                                  # one member with its own count
    hs = [HGP.from_hypergraph(hg, subrounds=s, seed=9) for hg, s in zip(hgs, subs)]
    b = Batch(hs)
    got = b.refine(3)
    for i, hg in enumerate(hgs):
        o = oracle.Oracle.from_hypergraph(hg, subrounds=subs[i], seed=9)
        want, _ = o.refine(3)
        assert np.array_equal(got[i][:, :5], want[:, :5])
        assert np.array_equal(hs[i].partition(), o.partition())
    b.close()
    for h, hg, s in zip(hs, hgs, subs):
        over = hg.part.copy()
        over[: max(1, hg.n * 2 // 3)] = 0
        h.set_partition(over)
        o = oracle.Oracle.from_hypergraph(hg, part=over, subrounds=s, seed=9)
        st, ph = h.rebalance(8)
        want, wph = o.rebalance(8)[:2]
        assert np.array_equal(st[:, :5], want[:, :5]) and np.array_equal(ph, wph)
        assert np.array_equal(h.partition(), o.partition())
        h.close()



@pytest.mark.parametrize("n,k,weighted", [(131_072, 64, False), (131_073, 7, True), (120_001, 17, True), (257, 64, True)])
@pytest.mark.parametrize("graph", [0, 1])
def test_largest_and_smallest_cluster_instances(n, k, weighted, graph):
    """At the line between one cluster and separate launches, saturated blocks among them; replayed
    as a graph too."""
    from paper_2010_10272_gb300 import HGP
    hg = synth.random_small(n + k, n, n, k, max_size=4, weighted=weighted, f=0.8, eps=0.01)   # 2.5 n pins
    o = oracle.Oracle.from_hypergraph(hg, subrounds=4, seed=9)
    want, _ = o.refine(6)
    h = HGP.from_hypergraph(hg, seed=9, graph=graph)
    got = np.concatenate([h.refine(3), h.refine(3)])
    assert np.array_equal(got[:, :5], want[:, :5])
    compare_state(h, o, check_phi=n < 1000)
    h.close()
