"""Handles created and dropped from several threads share the library's pinned
pages; each keeps its own counts (pytest -m gpu)."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_handles_from_threads():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2608_13144_gb300.lipcache import LipCache
    dev = torch.device("cuda", 0)
    rng = np.random.default_rng(0)
    W = torch.from_numpy(rng.standard_normal((4, 32)).astype(np.float32)).to(dev)
    b = torch.zeros(4, device=dev)
    rows = torch.from_numpy(rng.standard_normal((400, 32)).astype(np.float32)).to(dev)
    torch.cuda.synchronize()
    bad = []

    def work(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream(dev)):
                for r in range(6):
                    keep = [LipCache(32, 4, 400, device=dev) for _ in range(5)]  # more than a page in all threads
                    for j, c in enumerate(keep):
                        c.set_head(W, b)
                        n = 20 * (k + 1) + j
                        assert c.insert(rows[:n])[2] == n and c.size == n
                        assert (c.probe(rows[:n])[0].cpu().numpy() == np.arange(n)).all()
                    for c in keep:
                        c.close()
        except Exception as e:  # noqa: BLE001 (reported below)
            bad.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad[0]


def _pair(dev, n=2000, d=64, nq=300):
    from paper_2608_13144_gb300.lipcache import LipCache
    rng = np.random.default_rng(7)
    rows = rng.standard_normal((n, d)).astype(np.float32)
    Q = rng.standard_normal((nq, d)).astype(np.float32)
    dup = rng.random(nq) < 0.5
    Q[dup] = rows[rng.integers(0, n, dup.sum())] + np.float32(0.01) * rng.standard_normal((dup.sum(), d)).astype(np.float32)
    c = LipCache(d, 5, n, "tight", device=dev)
    c.set_head(torch.from_numpy((rng.standard_normal((5, d)) / 8).astype(np.float32)).to(dev), torch.zeros(5, device=dev))
    c.insert(torch.from_numpy(rows).to(dev))
    Qd = torch.from_numpy(Q).to(dev)
    ref = [t.cpu().numpy() for t in c.probe(Qd)]
    assert 0 < (ref[0] >= 0).sum() < nq
    return c, Qd, ref


def _out(B, dev):
    return (torch.empty(B, dtype=torch.int64, device=dev), torch.empty(B, dtype=torch.int32, device=dev),
            torch.empty(B, dtype=torch.float32, device=dev))


def _same(out, ref, k):
    for x, y in zip(ref, out):
        assert np.array_equal(x[:k].view(np.uint8), y.cpu().numpy().view(np.uint8)), k


def _hold(streams):
    """Make the streams wait for ~2 ms of work on another one, so that what is
    enqueued on them meanwhile starts together."""
    other = torch.cuda.Stream()
    with torch.cuda.stream(other):
        torch.cuda._sleep(4_000_000)
        e = other.record_event()
    for s in streams:
        s.wait_event(e)


@pytest.mark.parametrize("path", ["exact", "tensor"])
def test_probes_on_streams_that_nothing_orders(path):
    """Small probes finalize themselves by counting their CTAs. Probes of one
    handle that overlap on two streams may spoil each other's results, but
    nothing of it stays: every probe afterwards is right."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    dev = torch.device("cuda", 0)
    c, Q, ref = _pair(dev)
    c.set_probe_path(path)
    s = [torch.cuda.Stream(dev), torch.cuda.Stream(dev)]
    outs = [_out(Q.shape[0], dev), _out(70, dev)]
    torch.cuda.synchronize()
    for r in range(20):
        _hold(s)
        for _ in range(10):
            for k in range(2):
                with torch.cuda.stream(s[k]):
                    c.probe(Q[:outs[k][0].shape[0]], out=outs[k])
        torch.cuda.synchronize()
        for k in (300, 1, 129):
            out = _out(k, dev)
            out[0].fill_(-7)
            c.probe(Q[:k], out=out)
            _same(out, ref, k)
    c.close()


@pytest.mark.parametrize("path", ["exact", "tensor"])
def test_noalloc_beside_probe(path):
    """A no-allocation probe has scratch of its own, the counter too: it may
    run beside lipcache_probe on the same handle, called or replayed from a
    graph; so may a captured lipcache_probe, replayed after other probes."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    dev = torch.device("cuda", 0)
    c, Q, ref = _pair(dev)
    c.set_probe_path(path)
    s = [torch.cuda.Stream(dev), torch.cuda.Stream(dev)]
    a, b, g = _out(Q.shape[0], dev), _out(70, dev), _out(200, dev)
    c.probe_noalloc(Q[:70], b)  # (resolves the array's address before the capture)
    torch.cuda.synchronize()
    graph, own = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s[1]):
        c.probe_noalloc(Q[:70], b)
    with torch.cuda.graph(own, stream=s[1]):
        c.probe(Q[:200], out=g)
    for r in range(30):
        for t in a + b + g:
            t.fill_(-7)
        torch.cuda.synchronize()
        _hold(s)
        for _ in range(10):
            with torch.cuda.stream(s[0]):
                c.probe(Q, out=a)
            with torch.cuda.stream(s[1]):
                graph.replay() if r % 2 else c.probe_noalloc(Q[:70], b)
        torch.cuda.synchronize()
        _same(a, ref, Q.shape[0])
        _same(b, ref, 70)
        own.replay()
        torch.cuda.synchronize()
        _same(g, ref, 200)
    c.close()


def test_half_copy_leaves_memory():
    """The FP16 copy of the keys is only taken where it leaves three quarters of
    the free memory: a table of two fifths of the memory has none, a small one
    has. (Memory is reserved here, not written.)"""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2608_13144_gb300.lipcache import LipCache
    dev = torch.device("cuda", 0)
    LipCache(32, 4, 256, device=dev).close()  # the library's own memory
    torch.cuda.synchronize()
    torch.cuda.empty_cache()

    def taken(capacity):
        before = torch.cuda.mem_get_info(dev)[0]
        c = LipCache(32, 4, capacity, device=dev)
        after = torch.cuda.mem_get_info(dev)[0]
        c.close()
        return before - after

    per = 4 * 32 + 24  # bytes per entry, and 2 * 64 with the copy
    free = torch.cuda.mem_get_info(dev)[0]
    big = int(0.4 * free / per)
    assert taken(big) < per * big + (1 << 28)
    small = 1 << 20
    assert taken(small) >= (per + 128) * small
