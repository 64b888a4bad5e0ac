"""Nets of at most 4 pins in internal order keep no pin counts (Lambda, S1 and the size give them): every
reader and writer of the counts against the oracle, with few blocks (many movers per net) and many."""
import numpy as np
import pytest

import oracle
import synth
from parity_util import compare_state

pytestmark = pytest.mark.gpu
INTERNAL, LAUNCHES = 4, 32


@pytest.mark.parametrize("k", [2, 3, 32, 33, 64])
@pytest.mark.parametrize("max_size", [4, 7])
@pytest.mark.parametrize("variant", [{}, {"balance_moves": True}, {"revert_negative": True}])
def test_rounds(k, max_size, variant):
    from paper_2010_10272_gb300 import HGP
    hg = synth.random_small(k, 3001, 5003, k, max_size=max_size, weighted=True, f=0.9, eps=0.3)
    o = oracle.Oracle.from_hypergraph(hg, subrounds=1, seed=3, **variant)
    hs = [HGP.from_hypergraph(hg, subrounds=1, seed=3, debug=dbg, **variant) for dbg in (INTERNAL, INTERNAL | LAUNCHES)]
    for _ in range(4):
        want, _ = o.refine(1)
        for h in hs:
            assert np.array_equal(h.refine(1)[:, :5], want[:, :5])
            compare_state(h, o)
    rng = np.random.default_rng(k)
    u, part = rng.permutation(hg.n)[:900], o.partition()
    moves = np.stack([u, part[u], (part[u] + rng.integers(1, k, u.size)) % k], 1).astype(np.int32)
    for h in hs:
        assert np.array_equal(h.exact_gains(moves), o.exact_gains(moves))
        h.close()


def test_rebalancing_and_resume():
    from paper_2010_10272_gb300 import HGP
    hg = synth.random_small(5, 4000, 6000, 6, max_size=4, weighted=True, f=0.9)
    part = hg.part.copy()
    part[:2500] = 0
    h = HGP.from_hypergraph(hg, part=part, seed=3, debug=INTERNAL)
    o = oracle.Oracle.from_hypergraph(hg, part=part, seed=3)
    assert np.array_equal(h.rebalance(8)[0][:, :5], o.rebalance(8)[0])
    compare_state(h, o)
    h.refine(2)
    h2 = HGP.from_hypergraph(hg, part=part, seed=3, debug=INTERNAL | LAUNCHES)
    h2.import_state(h.export_state())
    assert np.array_equal(h2.refine(2), h.refine(2))
    o.refine(4)
    for x in (h, h2):
        compare_state(x, o)
        x.close()
