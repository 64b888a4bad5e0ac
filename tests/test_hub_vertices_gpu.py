"""Vertices of many nets beside vertices of few, numbered at random or by falling degree."""
import numpy as np
import pytest

import oracle
import synth
from parity_util import compare_state

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def hubs(seed, n, m, k, order="random", vertex_w=4, net_w=9, eps=0.1):
    """Nets of 2 to 7 pins, each pin the vertex of rank n x^5 for a uniform x (a few vertices are in a large
    part of all nets), ids by rank or at random."""
    rng = np.random.default_rng(seed)
    ids = np.arange(n) if order == "falling" else rng.permutation(n)
    nets = [np.unique(ids[np.minimum((n * rng.random(s) ** 5).astype(np.int64), n - 1)]) for s in rng.integers(2, 8, m)]
    hg = synth.random_small(seed, n, m, k, max_size=2, weighted=True, eps=eps)
    hg.net_off = np.concatenate([[0], np.cumsum([len(x) for x in nets])]).astype(hg.net_off.dtype)
    hg.pins = np.concatenate(nets).astype(np.int32)
    hg.vertex_w = rng.integers(1, vertex_w + 1, n).astype(np.int32) if vertex_w else None
    hg.net_w = rng.integers(1, net_w + 1, m).astype(np.int32) if net_w else None
    part = rng.integers(0, k, n).astype(np.int32)
    part[ids] = np.where(rng.random(n) < 0.7, np.arange(n) * k // n, part[ids])     # neighbours by rank together
    hg.part = part
    return hg


def degrees(hg):
    return np.bincount(hg.pins, minlength=hg.n)


@pytest.mark.parametrize("k", [2, 33, 64])
@pytest.mark.parametrize("order", ["random", "falling"])
@pytest.mark.parametrize("net_w", [0, 9, 3000])
def test_allocation_free_candidates(k, order, net_w):
    from paper_2010_10272_gb300.native import candidates_noalloc
    hg = hubs(k, 700, 6000, k, order, net_w=net_w)
    deg = degrees(hg)
    assert (deg > 96).sum() > 20 and (deg < 96).sum() > 300
    net = np.repeat(np.arange(hg.m, dtype=np.int32), np.diff(hg.net_off))
    dev = torch.device("cuda")
    args = [torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in
            (hg.net_off.astype(np.int32), hg.pins, np.concatenate([[0], np.cumsum(deg)]).astype(np.int32),
             net[np.argsort(hg.pins, kind="stable")])]
    part, vw = torch.from_numpy(hg.part).to(dev), torch.from_numpy(hg.vertex_w).to(dev)
    nw = torch.from_numpy(hg.net_w).to(dev) if net_w else None
    t = torch.empty(hg.n, dtype=torch.int32, device=dev)
    g = torch.empty(hg.n, dtype=torch.int64, device=dev)
    o = oracle.Oracle.from_hypergraph(hg, subrounds=2, seed=5)
    found = 0
    for s in range(2):
        assert candidates_noalloc(hg.n, hg.m, *args, k, hg.eps, part, t, g, vw, nw, subrounds=2, seed=5, s=s) == 0
        want_t, want_g = o.candidates(s)
        assert np.array_equal(t.cpu().numpy(), want_t) and np.array_equal(g.cpu().numpy(), want_g)
        found += (want_t[deg > 96] >= 0).sum()
    assert found > 0


@pytest.mark.parametrize("order", ["random", "falling"])
@pytest.mark.parametrize("n,m,k,count", [(60_000, 70_000, 5, 60_000), (60_000, 70_000, 40, 30_000), (900, 9000, 3, 800)])
def test_exact_gains(n, m, k, count, order):
    """Hubs among the few moves and among the many of a warp, in tables of half and of more than a
    million slots."""
    from paper_2010_10272_gb300 import HGP
    rng = np.random.default_rng(count)
    hg = hubs(n + k, n, m, k, order)
    u = rng.permutation(hg.n)[:count]
    hub = np.argsort(degrees(hg))[-40:]
    u = rng.permutation(np.unique(np.concatenate([u, hub])))
    a = hg.part[u]
    moves = np.stack([u, a, (a + rng.integers(1, k, u.size)) % k], 1).astype(np.int32)
    h = HGP.from_hypergraph(hg)
    assert np.array_equal(h.exact_gains(moves), oracle.Oracle.from_hypergraph(hg).exact_gains(moves))
    h.close()


@pytest.mark.parametrize("S", [1, 2, 3, 4, 16, 64])
@pytest.mark.parametrize("k,order", [(4, "falling"), (40, "falling"), (40, "random")])
def test_rebalancing(S, k, order):
    """Items of one to six segments, ending inside a tile's list, hubs side by side in the first."""
    from paper_2010_10272_gb300 import HGP
    hg = hubs(S + k, 9001, 14_000, k, order, eps=0.05)
    part = hg.part.copy()
    part[::3] = 0
    h = HGP.from_hypergraph(hg, part=part, subrounds=S, seed=2)
    o = oracle.Oracle.from_hypergraph(hg, part=part, subrounds=S, seed=2)
    st, ph = h.rebalance(8)
    want, wph = o.rebalance(8)[:2]
    assert np.array_equal(st[:, :5], want[:, :5]) and np.array_equal(ph, wph) and len(ph) > 0
    compare_state(h, o)
    h.close()


@pytest.mark.parametrize("k", [3, 32, 33, 64])
@pytest.mark.parametrize("net_w", [0, 2, 60, 800_000])
@pytest.mark.parametrize("variant", [{}, {"balance_moves": True}])
def test_rounds(k, net_w, variant):
    """Hubs whose nets weigh up to and more than 8191 (13 bit planes), by the cluster and by the launches."""
    from paper_2010_10272_gb300 import HGP
    hg = hubs(k, 700, 6000, k, "falling", net_w=net_w)
    net = np.repeat(np.arange(hg.m), np.diff(hg.net_off))
    W = np.bincount(hg.pins, weights=(hg.net_w if net_w else np.ones(hg.m))[net], minlength=hg.n)
    hub = degrees(hg) > 96
    assert (W[hub] <= 8191).any() or net_w > 60
    assert (W[hub] > 8191).any() == (net_w >= 60)
    o = oracle.Oracle.from_hypergraph(hg, subrounds=2, seed=9, **variant)
    want, _ = o.refine(3)
    for debug in (0, 32):
        h = HGP.from_hypergraph(hg, subrounds=2, seed=9, debug=debug, **variant)
        assert np.array_equal(h.refine(3)[:, :5], want[:, :5])
        compare_state(h, o)
        h.close()


@pytest.mark.parametrize("W", [8190, 8191, 8192])
@pytest.mark.parametrize("k", [2, 40])
def test_largest_sum_of_the_bit_planes(W, k):
    """One vertex whose W nets all reach one other block, at the last value the planes hold and beyond."""
    from paper_2010_10272_gb300 import HGP
    n = W + 200
    off = np.arange(0, 2 * W + 1, 2, dtype=np.int64)
    pins = np.stack([np.zeros(W, np.int32), np.arange(1, W + 1, dtype=np.int32)], 1).reshape(-1)
    part = np.zeros(n, np.int32)
    part[1:W + 1] = 1                          # every net of vertex 0 has its other pin there
    part[W + 1:] = 2 + np.arange(n - W - 1) % (k - 2) if k > 2 else 0
    vw = np.ones(n, np.int32)
    vw[W + 1:] = 2000                          # so that the block has room
    h = HGP(n, W, off, pins, k, 0.99, part, vw, subrounds=1, debug=32)
    o = oracle.Oracle(n, W, off, pins, k, 0.99, part, vw, subrounds=1)
    t, g = h.debug_candidates(0)
    want_t, want_g = o.candidates(0)
    assert np.array_equal(t, want_t) and np.array_equal(g, want_g)
    assert (t[0], g[0]) == (1, W)
    h.close()


@pytest.mark.parametrize("n,S", [(800_001, 1), (800_001, 3), (800_001, 4), (4_000_001, 4)])
def test_rebalancing_with_larger_items(n, S):
    """Items of up to 384 and 512 ids' active vertices: many vertices per warp (one CTA per SM)."""
    from paper_2010_10272_gb300 import HGP
    rng = np.random.default_rng(S)
    m, k = n // 4, 5
    pins = np.sort(rng.integers(0, n, (m, 3), dtype=np.int32), 1)
    pins = pins[(np.diff(pins, axis=1) > 0).all(1)]
    m = len(pins)
    off = np.arange(0, 3 * m + 1, 3, dtype=np.int64)
    part = rng.integers(0, k, n).astype(np.int32)
    part[rng.random(n) < 0.3] = 2
    args = (n, m, off, np.ascontiguousarray(pins.reshape(-1)), k, 0.03, part)
    h = HGP(*args, subrounds=S, apply_ctas_per_sm=1)
    o = oracle.Oracle(*args, subrounds=S)
    st, ph = h.rebalance(6)
    want, wph = o.rebalance(6)[:2]
    assert np.array_equal(st[:, :5], want[:, :5]) and np.array_equal(ph, wph)
    assert np.array_equal(h.partition(), o.partition())
    h.close()
