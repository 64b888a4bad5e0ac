"""The library's memory pool: memory whose release is pending, and memory used before."""
import gc

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _default_retention():
    from paper_2010_10272_gb300.native import set_pool_retention
    set_pool_retention(torch.cuda.mem_get_info()[1] // 64)


def test_create_waits_for_a_pending_release_on_another_stream():
    """On a nearly full device, a handle created while the rounds of a destroyed one still run takes
    that one's memory once it is released, instead of failing."""
    from paper_2010_10272_gb300 import HGP
    from paper_2010_10272_gb300.native import set_pool_retention
    n = m = 12_000_000                       # a handle of 1.1 GB, 0.6 more while it is created
    dev = torch.device("cuda")
    off = torch.arange(0, 4 * m + 1, 4, dtype=torch.int64, device=dev)
    step = torch.tensor([0, 7, 11, 19], device=dev)
    pins = ((torch.arange(m, device=dev)[:, None] + step) % n).sort(1)[0].to(torch.int32).reshape(-1).contiguous()
    part = (torch.arange(n, device=dev) % 16).to(torch.int32)
    try:
        set_pool_retention(0)
        a = HGP(n, m, off, pins, 16, 0.03, part, device=True, graph=1)
        want = a.refine(2)
        torch.cuda.synchronize()
        gc.collect()
        torch.cuda.empty_cache()
        rest = torch.empty(torch.cuda.mem_get_info()[0] - (850 << 20), dtype=torch.uint8, device=dev)
        a.refine(800, stats=False)           # one graph launch of about 0.4 s, still running below
        a.close()
        b = HGP(n, m, off, pins, 16, 0.03, part, device=True)
        assert np.array_equal(b.refine(2), want)
        b.close()
    finally:
        rest = None                          # noqa: F841
        torch.cuda.empty_cache()
        _default_retention()


def test_exact_gains_on_a_nearly_full_device():
    """16M incidences moved: with less free memory than the usual table takes, a smaller one is used."""
    from paper_2010_10272_gb300 import HGP
    from paper_2010_10272_gb300.native import set_pool_retention
    n = m = 4_000_000
    dev = torch.device("cuda")
    off = torch.arange(0, 4 * m + 1, 4, dtype=torch.int64, device=dev)
    step = torch.tensor([0, 7, 11, 19], device=dev)
    pins = ((torch.arange(m, device=dev)[:, None] + step) % n).sort(1)[0].to(torch.int32).reshape(-1).contiguous()
    part = (torch.arange(n, device=dev) % 16).to(torch.int32)
    u = np.random.default_rng(0).permutation(n)
    moves = np.stack([u, u % 16, (u + 5) % 16], 1).astype(np.int32)
    h = HGP(n, m, off, pins, 16, 0.03, part, device=True)
    try:
        set_pool_retention(0)
        want = h.exact_gains(moves)
        torch.cuda.synchronize()
        gc.collect()
        torch.cuda.empty_cache()
        rest = torch.empty(torch.cuda.mem_get_info()[0] - (1850 << 20), dtype=torch.uint8, device=dev)
        assert np.array_equal(h.exact_gains(moves), want)
    finally:
        rest = None                          # noqa: F841
        torch.cuda.empty_cache()
        _default_retention()
        h.close()


def test_a_handle_keeps_no_creation_scratch():
    """A handle made from device arrays of few nets and many vertices holds what its rounds use, not the
    buffers of its creation (8 bytes a vertex more)."""
    from paper_2010_10272_gb300 import HGP
    from paper_2010_10272_gb300.native import pool_usage
    n, m, k = 30_000_000, 1000, 8
    dev = torch.device("cuda")
    off = torch.arange(0, 64 * m + 1, 64, dtype=torch.int64, device=dev)
    pins = (torch.arange(m, device=dev)[:, None] * 29_000 + torch.arange(64, device=dev) * 400).to(torch.int32).reshape(-1)
    part = (torch.arange(n, device=dev) % k).to(torch.int32)
    before = pool_usage()[0]
    h = HGP(n, m, off, pins, k, 0.03, part, device=True)
    h.refine(1)
    torch.cuda.synchronize()
    kept = pool_usage()[0] - before
    tiles = -(-n // 2048)
    need = 4 * n + 2 * n + tiles * 2048 * (2 + 8) + 8 * k * tiles + 8 * k * 4096    # offsets, Pi twice, lists, candidates, ties
    assert need <= kept <= need + (64 << 20)
    h.close()


@pytest.mark.parametrize("skewed", [False, True])
def test_a_failed_creation_leaves_nothing(skewed):
    """Creations that run out of memory at one allocation or another free what they had."""
    from paper_2010_10272_gb300 import HGP, HGPError
    from paper_2010_10272_gb300.native import pool_usage, set_pool_retention
    n = m = 4_000_000
    dev = torch.device("cuda")
    size = torch.full((m,), 4, dtype=torch.int64, device=dev)
    first = torch.arange(m, device=dev)
    if skewed:                                # large nets: internal order
        size[:40] = 100_000
    off = torch.zeros(m + 1, dtype=torch.int64, device=dev)
    off[1:] = torch.cumsum(size, 0)
    net = torch.repeat_interleave(first, size)
    pins = (torch.clamp(net, max=n - 100_000) + torch.arange(net.numel(), device=dev) - off[net]).to(torch.int32)
    part = (torch.arange(n, device=dev) % 16).to(torch.int32)
    del net, size, first
    failed = 0
    try:
        set_pool_retention(0)
        for free_mb in list(range(60, 700, 40)) + [1500]:
            torch.cuda.synchronize()
            torch.cuda.empty_cache()
            before = pool_usage()[0]
            rest = torch.empty(torch.cuda.mem_get_info()[0] - (free_mb << 20), dtype=torch.uint8, device=dev)
            try:
                HGP(n, m, off, pins, 16, 0.03, part, device=True).close()
            except HGPError as e:
                assert e.code == 2
                failed += 1
            torch.cuda.synchronize()
            assert pool_usage()[0] == before, free_mb
            del rest
        assert 3 <= failed <= 16
    finally:
        rest = None                          # noqa: F841
        torch.cuda.empty_cache()
        _default_retention()
