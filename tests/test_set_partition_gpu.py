"""A partition's state (Phi, Lambda, objective, block weights) built from scratch, against the oracle's."""
import numpy as np
import pytest

import oracle
import synth
from parity_util import compare_state

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("phi_width", [0, 1, 2, 4])
@pytest.mark.parametrize("k", [2, 5, 32, 33, 64])
@pytest.mark.parametrize("sizes", ["tiny", "mixed", "big"])
def test_state_of_a_new_partition(phi_width, k, sizes):
    """Groups of 32 nets of at most 4 pins (a lane each), larger ones (walked flattened), and nets beyond
    a 1-byte entry (255) or 2048 pins (a CTA each); rows that are no multiple of 16 bytes; the last
    group partly empty."""
    from paper_2010_10272_gb300 import HGP
    rng = np.random.default_rng(k)
    n, m = 5003, 1037
    size = rng.integers(0, 5, m) if sizes == "tiny" else rng.integers(0, 40, m)
    if sizes == "big":
        size[[3, 40, 41, 700]] = [255, 256, 2048, 2049]
        size[m - 1] = n
    pins = np.concatenate([np.sort(rng.choice(n, s, replace=False)) for s in size]).astype(np.int32)
    off = np.concatenate([[0], np.cumsum(size)]).astype(np.int64)
    vw = rng.integers(1, 2**20, n).astype(np.int32) if k == 5 else None
    nw = rng.integers(1, 9, m).astype(np.int32) if k != 2 else None
    first, second = rng.integers(0, k, (2, n)).astype(np.int32)
    h = HGP(n, m, off, pins, k, 0.03, first, vw, nw, phi_width=phi_width)
    compare_state(h, oracle.Oracle(n, m, off, pins, k, 0.03, first, vw, nw))
    h.refine(2)
    with pytest.raises(Exception):                      # refused, and the state stays
        h.set_partition(np.where(np.arange(n) == n - 1, k, second))
    o = oracle.Oracle(n, m, off, pins, k, 0.03, first, vw, nw)
    o.refine(2)
    compare_state(h, o)
    for device in (False, True):
        h.set_partition(torch.from_numpy(second).cuda() if device else second, device=device)
        o = oracle.Oracle(n, m, off, pins, k, 0.03, second, vw, nw)
        compare_state(h, o)
        assert np.array_equal(h.refine(2)[:, :5], o.refine(2)[0])
    h.close()


@pytest.mark.parametrize("debug", [0, 2, 4, 6])
@pytest.mark.parametrize("where", ["first", "middle", "last"])
def test_pin_order_is_checked_wherever_it_breaks(debug, where):
    """A repeated or falling pin inside a net is refused, a falling step between two nets is not; with
    empty nets, nets of one pin and a net of 100,000 among them, on every creation path."""
    from paper_2010_10272_gb300 import HGP, HGPError
    rng = np.random.default_rng(3)
    n = 120_000
    size = rng.integers(0, 4, 30_000)
    size[17_000] = 100_000
    size[20_000] = 9_000
    pins = np.concatenate([np.sort(rng.choice(n, s, replace=False)) for s in size]).astype(np.int32)
    off = np.concatenate([[0], np.cumsum(size)]).astype(np.int64)
    part = rng.integers(0, 9, n).astype(np.int32)
    h = HGP(n, size.size, off, pins, 9, 0.03, part, debug=debug)
    compare_state(h, oracle.Oracle(n, size.size, off, pins, 9, 0.03, part))
    h.close()
    at = {"first": off[np.flatnonzero(size >= 2)[0]], "middle": off[17_000] + 50_000,
          "last": off[np.flatnonzero(size >= 2)[-1]]}[where]
    for delta in (0, 1):
        bad = pins.copy()
        bad[at + 1] = bad[at] - delta
        for device in (False, True):
            a = [torch.from_numpy(x).cuda() if device else x for x in (off, bad, part)]
            with pytest.raises(HGPError) as ei:
                HGP(n, size.size, a[0], a[1], 9, 0.03, a[2], debug=debug, device=device)
            assert ei.value.code == 1
