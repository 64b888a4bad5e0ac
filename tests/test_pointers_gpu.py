"""Device arrays of the caller, wherever they are."""
import numpy as np
import pytest

import oracle
import synth
from parity_util import compare_state

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _allocated(kind, values):
    """An int32 array in device memory at the end of its allocation, in managed or in page-locked host
    memory: (address, owner)."""
    import ctypes
    rt = ctypes.CDLL("libcudart.so.%d" % int(torch.version.cuda.split(".")[0]))
    p, nbytes = ctypes.c_void_p(), values.nbytes
    room = -(-nbytes // (2 << 20)) * (2 << 20)
    call = {"device": rt.cudaMalloc, "managed": rt.cudaMallocManaged, "pinned": rt.cudaMallocHost}[kind]
    args = (ctypes.c_uint(1),) if kind == "managed" else ()
    assert call(ctypes.byref(p), ctypes.c_size_t(room), *args) == 0
    at = p.value + room - nbytes
    assert rt.cudaMemcpy(ctypes.c_void_p(at), values.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(nbytes), 4) == 0
    return at, lambda: (rt.cudaFreeHost if kind == "pinned" else rt.cudaFree)(p)


@pytest.mark.parametrize("kind", ["device", "managed", "pinned"])
def test_device_partition_wherever_it_is(kind):
    from paper_2010_10272_gb300 import HGP
    hg = synth.random_small(4, 5003, 4000, 6, max_size=7)
    second = np.random.default_rng(1).integers(0, 6, hg.n).astype(np.int32)
    at, free = _allocated(kind, second)
    h = HGP.from_hypergraph(hg)
    h.set_partition(at, device=True)
    compare_state(h, oracle.Oracle.from_hypergraph(hg, part=second))
    h.close()
    free()


@pytest.mark.parametrize("kind", ["device", "managed", "pinned"])
def test_allocation_free_offsets_wherever_they_are(kind):
    from paper_2010_10272_gb300 import HGP
    from paper_2010_10272_gb300.native import candidates_noalloc
    hg = synth.random_small(4, 5003, 4000, 6, max_size=7)
    net = np.repeat(np.arange(hg.m, dtype=np.int32), np.diff(hg.net_off))
    voff = np.concatenate([[0], np.cumsum(np.bincount(hg.pins, minlength=hg.n))]).astype(np.int32)
    pins, voff, inc, part = (torch.from_numpy(x).cuda() for x in
                             (hg.pins, voff, net[np.argsort(hg.pins, kind="stable")], hg.part))
    t = torch.empty(hg.n, dtype=torch.int32, device="cuda")
    g = torch.empty(hg.n, dtype=torch.int64, device="cuda")
    off, free = _allocated(kind, hg.net_off.astype(np.int32))
    assert candidates_noalloc(hg.n, hg.m, off, pins, voff, inc, hg.k, hg.eps, part, t, g) == 0
    assert candidates_noalloc(hg.n, hg.m, off, None, voff, None, hg.k, hg.eps, part, t, g) == 1
    h = HGP.from_hypergraph(hg)
    want_t, want_g = h.debug_candidates(0)
    assert np.array_equal(t.cpu().numpy(), want_t) and np.array_equal(g.cpu().numpy(), want_g)
    h.close()
    free()
