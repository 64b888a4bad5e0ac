"""Contraction of nets whose fingerprints agree in the bits that their table slot keeps."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")


def _splitmix(z):
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _fingerprints(pins):
    """64-bit fingerprints of two-pin nets (uint64 [count, 2])."""
    x = (pins + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
    x = (x ^ (x >> np.uint64(32))) * np.uint64(0xD1342543DE82EF95)
    x ^= x >> np.uint64(32)
    return _splitmix(x.sum(1, dtype=np.uint64) ^ (np.uint64(2) << np.uint64(32)))


def shared_slots(n, count):
    """Pairs of two-pin nets that agree in the upper 32 and the lower 10 bits of their fingerprints: in a
    table of 1024 slots they start at the same one and share it."""
    rng = np.random.default_rng(2)
    u = rng.integers(0, n, count).astype(np.uint64)
    v = rng.integers(0, n - 1, count).astype(np.uint64)
    v += v >= u
    pins = np.stack([np.minimum(u, v), np.maximum(u, v)], 1)
    pins = np.unique(pins[:, 0] * np.uint64(n) + pins[:, 1])
    pins = np.stack([pins // np.uint64(n), pins % np.uint64(n)], 1)
    key = _fingerprints(pins)
    slot = (key >> np.uint64(32) << np.uint64(10)) | (key & np.uint64(1023))
    order = np.argsort(slot, kind="stable")
    same = np.flatnonzero(slot[order][1:] == slot[order][:-1])
    return pins[order[same]].astype(np.int32), pins[order[same + 1]].astype(np.int32), key[order[same]], key[order[same + 1]]


@pytest.mark.gpu
def test_nets_that_share_a_slot():
    from paper_2010_10272_gb300 import Coarse
    n = 30_000
    a, b, ka, kb = shared_slots(n, 12_000_000)
    assert len(a) >= 8 and (ka != kb).all()
    a, b = a[:100], b[:100]
    rng = np.random.default_rng(5)
    nets = np.concatenate([a, b, b, a, a])                          # two nets, three and two times each
    nets = nets[rng.permutation(len(nets))]
    assert len(nets) <= 768                                         # a table of 1024 slots
    off = np.arange(0, 2 * len(nets) + 1, 2, dtype=np.int64)
    pins = np.ascontiguousarray(nets.reshape(-1))
    nw = rng.integers(1, 9, len(nets)).astype(np.int32)
    cluster = np.arange(n, dtype=np.int32)
    d = [torch.from_numpy(x).cuda() for x in (off, pins, nw, cluster)]
    c = Coarse(n, len(nets), d[0], d[1], None, d[2], d[3])
    got = c.to_host()
    want = oracle.contract(n, len(nets), off, pins, None, nw, cluster)
    assert got["m"] == want["m"] == 2 * len(a)
    for key in ("net_off", "pins", "vertex_w", "net_w", "map"):
        np.testing.assert_array_equal(got[key], want[key], err_msg=key)
    c.close()
