"""Every entry point on memory that the pool kept from other work."""
import numpy as np
import pytest

import oracle
import synth
from parity_util import compare_state

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def kept():
    """The pool keeps what was freed, among it arrays of other values."""
    from paper_2010_10272_gb300 import HGP
    from paper_2010_10272_gb300.native import pool_usage, set_pool_retention
    set_pool_retention(1 << 40)               # whatever else is alive
    hg = synth.random_small(1, 400_000, 300_000, 64, max_size=9, weighted=True)
    hs = [HGP.from_hypergraph(hg, revert_negative=True) for _ in range(2)]
    for h in hs:
        h.refine(2)
        h.close()
    torch.cuda.synchronize()
    assert pool_usage()[1] > 100 << 20
    yield
    set_pool_retention(torch.cuda.mem_get_info()[1] // 64)


@pytest.mark.parametrize("k,debug", [(5, 0), (5, 2 | 32), (40, 4), (64, 4 | 32)])
@pytest.mark.parametrize("variant", [{}, {"revert_negative": True}])
@pytest.mark.parametrize("device", [False, True])
def test_handles(k, debug, variant, device):
    from paper_2010_10272_gb300 import HGP
    hg = synth.random_small(k, 30_001, 25_000, k, max_size=7, weighted=True, eps=0.1)
    a = [hg.net_off, hg.pins, hg.part, hg.vertex_w, hg.net_w]
    if device:
        a = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in a]
    h = HGP(hg.n, hg.m, a[0], a[1], k, hg.eps, a[2], a[3], a[4], debug=debug, device=device, **variant)
    o = oracle.Oracle.from_hypergraph(hg, **variant)
    assert np.array_equal(h.refine(3)[:, :5], o.refine(3)[0][:, :5])
    compare_state(h, o)
    rng = np.random.default_rng(k)
    u, part = rng.permutation(hg.n)[:3000], o.partition()
    moves = np.stack([u, part[u], (part[u] + rng.integers(1, k, u.size)) % k], 1).astype(np.int32)
    assert np.array_equal(h.exact_gains(moves), o.exact_gains(moves))
    h.close()


@pytest.mark.parametrize("sizes", [(0, 9), (0, 700), (0, 12_000)])
def test_contraction(sizes):
    from paper_2010_10272_gb300 import Coarse
    rng = np.random.default_rng(sizes[1])
    n = 20_000
    nets = [np.sort(rng.choice(n, s, replace=False)) for s in rng.integers(*sizes, 200)]
    nets += nets[:50]
    off = np.concatenate([[0], np.cumsum([len(x) for x in nets])]).astype(np.int64)
    pins = np.concatenate(nets).astype(np.int32)
    cluster = rng.integers(0, n // 3, n).astype(np.int32)
    d = [torch.from_numpy(x).cuda() for x in (off, pins, cluster)]
    c = Coarse(n, len(nets), d[0], d[1], None, None, d[2])
    got, want = c.to_host(), oracle.contract(n, len(nets), off, pins, None, None, cluster)
    for key in ("n", "m", "net_off", "pins", "vertex_w", "net_w", "map"):
        np.testing.assert_array_equal(got[key], want[key], err_msg=key)
    c.close()
