"""The arrays of a Coarse after its stream is gone."""
import ctypes

import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _contract(hg, cluster, stream):
    from paper_2010_10272_gb300 import Coarse
    d = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (hg.net_off.astype(np.int64), hg.pins, cluster)]
    return Coarse(hg.n, hg.m, d[0], d[1], None, None, d[2], stream=stream)


def test_released_after_its_stream_was_destroyed():
    """The memory comes back: 40 coarse hypergraphs of 40 MB, released after their streams, leave no more
    than the first of them in use."""
    from paper_2010_10272_gb300.native import set_pool_retention
    rt = ctypes.CDLL("libcudart.so.%d" % int(torch.version.cuda.split(".")[0]))
    rng = np.random.default_rng(0)
    hg = synth.random_small(11, 2_000_000, 1_200_000, 2, max_size=6)
    cluster = rng.integers(0, hg.n // 2, hg.n).astype(np.int32)
    set_pool_retention(0)
    try:
        free = []
        for i in range(40):
            st = ctypes.c_void_p()
            assert rt.cudaStreamCreate(ctypes.byref(st)) == 0
            c = _contract(hg, cluster, st.value)
            if i == 0:
                got = c.to_host()
                want = oracle.contract(hg.n, hg.m, hg.net_off, hg.pins, None, None, cluster)
                for key in ("net_off", "pins", "vertex_w", "net_w", "map"):
                    np.testing.assert_array_equal(got[key], want[key], err_msg=key)
            assert rt.cudaStreamDestroy(st) == 0
            c.close()
            torch.cuda.synchronize()
            free.append(torch.cuda.mem_get_info()[0])
        assert min(free[1:]) >= free[0] - (64 << 20)
    finally:
        set_pool_retention(torch.cuda.mem_get_info()[1] // 64)


def test_released_arrays_are_the_pools_again():
    from paper_2010_10272_gb300.native import pool_usage, set_pool_retention
    set_pool_retention(1 << 40)
    hg = synth.random_small(12, 200_000, 120_000, 2, max_size=6)
    cluster = (np.arange(hg.n) // 2).astype(np.int32)
    before = pool_usage()[0]
    c = _contract(hg, cluster, None)
    live = pool_usage()[0] - before
    assert live > 4 * c.num_pins
    c.close()
    used, kept = pool_usage()
    assert used == before and kept >= live
    set_pool_retention(torch.cuda.mem_get_info()[1] // 64)
