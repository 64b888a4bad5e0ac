"""Exact gains where the work of a warp changes: few and many moves, vertices of few and of many nets."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,k", [(40, 30, 2), (300, 6000, 5), (20_000, 3_000, 33), (3000, 9000, 64)])
@pytest.mark.parametrize("count", [1, 31, 33, 4000])
def test_counts_and_degrees(n, m, k, count):
    from paper_2010_10272_gb300 import HGP
    rng = np.random.default_rng(count)
    hg = synth.random_small(n + m, max(n, k), m, k, max_size=7, weighted=True)
    u = rng.permutation(hg.n)[:count]
    a = hg.part[u]
    moves = np.stack([u, a, (a + rng.integers(1, k, u.size)) % k], 1).astype(np.int32)
    h = HGP.from_hypergraph(hg)
    o = oracle.Oracle.from_hypergraph(hg)
    assert np.array_equal(h.exact_gains(moves), o.exact_gains(moves))
    h.close()


@pytest.mark.parametrize("n,m,k", [(40_000, 30_000, 7), (70_000, 160_000, 40)])
@pytest.mark.parametrize("count", [4863, 9728, 34_047])
def test_moves_of_one_warp(n, m, k, count):
    """One move, a few, and many moves of a warp; tables at most half and at most two thirds full."""
    from paper_2010_10272_gb300 import HGP
    rng = np.random.default_rng(count)
    hg = synth.random_small(n + m, n, m, k, max_size=12, weighted=True)
    u = rng.permutation(hg.n)[:count]
    a = hg.part[u]
    moves = np.stack([u, a, (a + rng.integers(1, k, u.size)) % k], 1).astype(np.int32)
    h = HGP.from_hypergraph(hg)
    o = oracle.Oracle.from_hypergraph(hg)
    assert np.array_equal(h.exact_gains(moves), o.exact_gains(moves))
    h.close()
