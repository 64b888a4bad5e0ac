"""Contraction at the edges of its net size classes (a lane, a warp with 1 to 16 values per lane, a CTA,
merged 2048-pin chunks), with identical nets among them, against the oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("factor", [1, 2, 60])
@pytest.mark.parametrize("order", ["shuffled", "falling"])
def test_class_edges(factor, order):
    from paper_2010_10272_gb300 import Coarse
    rng = np.random.default_rng(factor)
    n = 30_000
    edges = [8, 32, 64, 128, 256, 512, 2048, 4096, 8192, 16_384]
    size = np.concatenate([[x - 1, x, x + 1] for x in edges] + [[0, 0, 1, 2, 3, 20_001, n], rng.integers(0, 700, 300)])
    size = rng.permutation(size) if order == "shuffled" else np.sort(size)[::-1]
    nets = [np.sort(rng.choice(n, s, replace=False)) for s in size]
    nets = [nets[i] for i in rng.permutation(np.r_[0:len(nets), 0:len(nets):3])]      # a third of them twice
    off = np.concatenate([[0], np.cumsum([len(x) for x in nets])]).astype(np.int64)
    pins = np.concatenate(nets).astype(np.int32)
    vw = rng.integers(1, 5, n).astype(np.int32)
    nw = rng.integers(1, 9, len(nets)).astype(np.int32)
    cluster = rng.integers(0, max(1, n // factor), n).astype(np.int32) if factor > 1 else rng.permutation(n).astype(np.int32)
    d = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (off, pins, vw, nw, cluster)]
    for _ in range(2):                                                                # the second reuses the pool's memory
        c = Coarse(n, len(nets), *d)
        got = c.to_host()
        want = oracle.contract(n, len(nets), off, pins, vw, nw, cluster)
        assert (got["n"], got["m"]) == (want["n"], want["m"])
        for key in ("net_off", "pins", "vertex_w", "net_w", "map"):
            np.testing.assert_array_equal(got[key], want[key], err_msg=key)
        c.close()
