"""The serving loop's default memory budget."""
import pytest

torch = pytest.importorskip("torch")


def test_what_the_pool_keeps_is_free_for_requests(monkeypatch):
    from paper_2010_10272_gb300 import serve
    monkeypatch.setattr(torch.cuda, "mem_get_info", lambda *a: (10 << 30, 16 << 30))
    monkeypatch.setattr(torch.cuda, "is_available", lambda: True)
    monkeypatch.setattr(serve, "pool_usage", lambda: (1 << 30, 3 << 30), raising=False)
    assert serve.Server(reserve_bytes=1 << 30, creators=0).memory_budget == 12 << 30
    assert serve.Server(memory_budget=5, creators=0).memory_budget == 5


@pytest.mark.gpu
def test_pool_usage():
    import synth
    from paper_2010_10272_gb300 import HGP
    from paper_2010_10272_gb300.native import pool_usage, set_pool_retention
    set_pool_retention(1 << 40)
    hg = synth.random_small(3, 300_000, 200_000, 8, max_size=6)
    before = pool_usage()[0]
    h = HGP.from_hypergraph(hg)
    live = pool_usage()[0] - before
    assert live > 20 * hg.n
    h.close()
    torch.cuda.synchronize()
    used, kept = pool_usage()
    assert used == before and kept >= live
    set_pool_retention(torch.cuda.mem_get_info()[1] // 64)


@pytest.mark.gpu
@pytest.mark.parametrize("n,m,k,weighted", [(3000, 2000, 2, False), (200_000, 150_000, 40, True), (1_500_000, 1_100_000, 16, True)])
def test_estimate_covers_a_handle(n, m, k, weighted):
    import synth
    from paper_2010_10272_gb300 import HGP
    from paper_2010_10272_gb300.native import pool_usage
    from paper_2010_10272_gb300.serve import estimate_device_bytes
    hg = synth.random_small(n, n, m, k, max_size=6, weighted=weighted)
    before = pool_usage()[0]
    h = HGP.from_hypergraph(hg)
    h.refine(1)
    assert pool_usage()[0] - before <= estimate_device_bytes(n, m, int(hg.net_off[-1]), k, 6, weighted, weighted)
    h.close()
