"""hgp_candidates_noalloc where its paths part: nets read by a lane or by a warp, W(u) in 6 or 11 bit
planes or beyond them, ranges that end inside a warp; lists out of order at their edges."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _csr(hg):
    net = np.repeat(np.arange(hg.m, dtype=np.int32), np.diff(hg.net_off))
    order = np.argsort(hg.pins, kind="stable")
    off = np.concatenate([[0], np.cumsum(np.bincount(hg.pins, minlength=hg.n))]).astype(np.int32)
    return hg.net_off.astype(np.int32), hg.pins, off, net[order]


@pytest.mark.parametrize("n,m,max_size,scale", [(1, 1, 1, 1), (127, 300, 16, 1), (129, 900, 17, 9), (5000, 4000, 40, 1),
                                                (400, 4000, 9, 30), (300, 60, 300, 1)])
@pytest.mark.parametrize("k", [2, 33, 64])
def test_candidates_equal_the_handle(n, m, max_size, scale, k):
    from paper_2010_10272_gb300 import HGP
    from paper_2010_10272_gb300.native import candidates_noalloc
    n = max(n, k)
    hg = synth.random_small(n + k, n, m, k, max_size=max_size, weighted=True, f=0.8, eps=0.1)
    hg.net_w = (hg.net_w * scale).astype(np.int32)
    dev = torch.device("cuda")
    args = [torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in _csr(hg)]
    part, vw, nw = (torch.from_numpy(x).to(dev) for x in (hg.part, hg.vertex_w, hg.net_w))
    t = torch.empty(n, dtype=torch.int32, device=dev)
    g = torch.empty(n, dtype=torch.int64, device=dev)
    h = HGP.from_hypergraph(hg, subrounds=3, seed=5)
    for s in range(3):
        assert candidates_noalloc(n, hg.m, *args, k, hg.eps, part, t, g, vw, nw, subrounds=3, seed=5, s=s) == 0
        want_t, want_g = h.debug_candidates(s)
        assert np.array_equal(t.cpu().numpy(), want_t) and np.array_equal(g.cpu().numpy(), want_g)
    h.close()


def test_falling_entries_are_refused():
    from paper_2010_10272_gb300.native import candidates_noalloc
    hg = synth.random_small(3, 500, 400, 4, max_size=8)
    dev = torch.device("cuda")
    off, pins, voff, inc = _csr(hg)
    part = torch.from_numpy(hg.part).to(dev)
    t = torch.full((500,), 77, dtype=torch.int32, device=dev)
    g = torch.empty(500, dtype=torch.int64, device=dev)

    def call(p, i):
        a = [torch.from_numpy(x).to(dev) for x in (off, p, voff, i)]
        return candidates_noalloc(500, hg.m, *a, 4, 0.03, part, t, g)
    for lists, which in ((np.diff(off), 0), (np.diff(voff), 1)):
        for at in np.flatnonzero(lists >= 2)[[0, -1]]:
            b = (off, voff)[which][at]
            x = [pins.copy(), inc.copy()]
            x[which][[b, b + 1]] = x[which][[b + 1, b]]
            assert call(*x) == 1
            x[which][b] = x[which][b + 1]
            assert call(*x) == 1
    assert bool((t == 77).all())                       # nothing was written by a refused call
    assert call(pins, inc) == 0
