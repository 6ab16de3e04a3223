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
