"""The kernels of a round at the sizes where their tiling can go wrong, against the oracle (exact)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _check(hg, rounds=4, subrounds=4, eps=None, **kw):
    from paper_2010_10272_gb300 import HGP
    if eps is not None:
        hg.eps = eps
    h = HGP.from_hypergraph(hg, subrounds=subrounds, seed=9, **kw)
    o = oracle.Oracle.from_hypergraph(hg, subrounds=subrounds, seed=9)
    want, _ = o.refine(rounds)
    got = h.refine(rounds)
    assert np.array_equal(got[:, :5], want[:, :5])
    assert np.array_equal(h.partition(), o.partition())
    assert h.objective() == o.objective() == h.objective_from_phi()
    h.close()


@pytest.mark.parametrize("n", [2047, 2048, 2049, 4096, 6145, 33_000])
@pytest.mark.parametrize("weighted", [False, True])
def test_ties_at_the_threshold_gain(n, weighted):
    """Small nets give few distinct gains, so a saturated block's budget ends inside a long run of
    equal gains: the last approved id falls anywhere in a tile of 2048 vertices."""
    hg = synth.random_small(n, n, n, 5, max_size=3, weighted=weighted, f=0.9)
    _check(hg, eps=0.004)
    _check(hg, eps=0.004, subrounds=1)
