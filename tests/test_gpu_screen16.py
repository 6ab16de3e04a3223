"""The FP16 screen of the tensor probe against the exact kernel, bit for bit:
widths around its 64-feature chunks and 16-feature MMA steps, alignments,
every way a table grows, and what falls back to TF32 (pytest -m gpu)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    return torch.device("cuda", 0)


def make(dev, d, C, rows, scale=1.0, capacity=None):
    from paper_2608_13144_gb300.lipcache import LipCache
    rng = np.random.default_rng(d * 31 + C)
    W = (rng.standard_normal((C, d)) / np.sqrt(d)).astype(np.float32) / np.float32(scale)
    c = LipCache(d, C, capacity or len(rows), "tight", device=dev)
    c.set_head(torch.from_numpy(W).to(dev), torch.zeros(C, device=dev))
    return c


def same_as_exact(c, Q, paths, need_hits=True):
    c.set_probe_path("exact")
    ref = [t.cpu().numpy() for t in c.probe(Q)]
    if need_hits:
        assert (ref[0] >= 0).any() and (Q.shape[1] == 1 or (ref[0] < 0).any())
    for path in paths:
        c.set_probe_path(path)
        got = [t.cpu().numpy() for t in c.probe(Q)]
        assert c.info()["device_errors"] == 0
        for x, y in zip(ref, got):
            assert np.array_equal(x.view(np.uint8), y.view(np.uint8)), path
    return ref


def data(rng, n, d, nq, noise=0.01):
    rows = rng.standard_normal((n, d)).astype(np.float32)
    Q = rng.standard_normal((nq, d)).astype(np.float32)
    dup = rng.random(nq) < 0.5
    Q[dup] = rows[rng.integers(0, n, dup.sum())] + noise * rng.standard_normal((dup.sum(), d)).astype(np.float32)
    return rows, Q


@pytest.mark.parametrize("d", [1, 15, 16, 17, 63, 64, 65, 80, 128, 129, 192, 250, 256])
def test_widths(dev, d):
    rng = np.random.default_rng(d)
    rows, Q = data(rng, 3001, d, 257)
    c = make(dev, d, 5, rows)
    c.insert(torch.from_numpy(rows).to(dev))
    paths = ["tensor", "tensor_single", "tensor_pair"]
    same_as_exact(c, torch.from_numpy(Q).to(dev), paths)
    # a batch that is not 16-byte aligned: the recheck reads it in place
    buf = torch.zeros(Q.size + 1, device=dev)
    buf[1:] = torch.from_numpy(Q.reshape(-1))
    same_as_exact(c, buf[1:].view(Q.shape), paths)
    c.close()


@pytest.mark.parametrize("d,n,nq", [(257, 9001, 129), (300, 40000, 64), (448, 20001, 300), (449, 20001, 300),
                                    (512, 30000, 1000)])
def test_wide_auto(dev, d, n, nq):
    """d in (256, 512]: "auto" screens in FP16 from 2^24 multiply-adds on; the
    named tensor paths stay refused."""
    from paper_2608_13144_gb300 import LipCacheError
    rng = np.random.default_rng(d + n)
    rows, Q = data(rng, n, d, nq)
    c = make(dev, d, 4, rows)
    c.insert(torch.from_numpy(rows).to(dev))
    same_as_exact(c, torch.from_numpy(Q).to(dev), ["auto"])
    assert c.info()["last_probe_path"] in (3, 4)
    with pytest.raises(LipCacheError):
        c.set_probe_path("tensor")
    c.close()


@pytest.mark.parametrize("n,nq", [(40, 1), (255, 128), (256, 129), (513, 4096), (200_000, 1025)])
def test_sizes(dev, n, nq):
    """One tile, an odd last tile, ragged queries, long ranges (stages released
    in pairs with one chunk per tile)."""
    rng = np.random.default_rng(n)
    rows, Q = data(rng, n, 48, nq)
    c = make(dev, 48, 5, rows)
    c.insert(torch.from_numpy(rows).to(dev))
    same_as_exact(c, torch.from_numpy(Q).to(dev), ["tensor", "tensor_pair"], need_hits=n > 1000)
    c.close()


@pytest.mark.parametrize("grow", ["unaligned", "async", "select", "kcenter", "writeback"])
@pytest.mark.parametrize("d", [33, 96])
def test_growth(dev, grow, d):
    """Every path that appends entries writes their FP16 copies."""
    rng = np.random.default_rng(d)
    rows, Q = data(rng, 3000, d, 500)
    c = make(dev, d, 6, rows)
    R = torch.from_numpy(rows).to(dev)
    if grow == "unaligned":
        buf = torch.zeros(rows.size + 1, device=dev)
        buf[1:] = R.reshape(-1)
        c.insert(buf[1:].view(rows.shape))
    elif grow == "async":
        for k in range(0, 3000, 700):
            c.insert(R[k:k + 700], wait=False)
    elif grow == "select":
        c.insert_select(R, strategy="radius_dedup", budget_total=2500)
    elif grow == "kcenter":
        c.insert_select(R, strategy="kcenter", budget_per_class=300)
    else:
        c.insert(R[:1000])
        c.probe_writeback(R[1000:])
    same_as_exact(c, torch.from_numpy(Q).to(dev), ["tensor", "tensor_pair"])
    c.close()


@pytest.mark.parametrize("n", [1, 255, 256, 257, 700])
@pytest.mark.parametrize("how", ["insert", "select", "kcenter"])
def test_rows_past_the_end(dev, how, n):
    """The table's memory is not cleared at creation: the rows past the last
    entry of its tile are zero because appending entries clears them, so
    memory full of infinities (as FP16 and as FP32) left by another owner
    neither reaches a result nor makes candidates of the pairs with it."""
    from paper_2608_13144_gb300.lipcache import LipCache
    junk = [torch.full((64, 1024, 1024), torch.inf, device=dev) for _ in range(4)]
    del junk
    torch.cuda.empty_cache()  # the next allocations may get this memory
    rng = np.random.default_rng(n)
    rows, Q = data(rng, n, 32, 300)
    c = LipCache(32, 4, 200_000, "tight", device=dev)
    c.set_head(torch.from_numpy((rng.standard_normal((4, 32)) / 6).astype(np.float32)).to(dev), torch.zeros(4, device=dev))
    R = torch.from_numpy(rows).to(dev)
    if how == "insert":
        c.insert(R)
    else:
        c.insert_select(R, strategy="radius_dedup" if how == "select" else "kcenter",
                        budget_per_class=0 if how == "select" else 400)
    Qd = torch.from_numpy(Q).to(dev)
    same_as_exact(c, Qd, ["tensor", "tensor_pair"], need_hits=False)
    c.set_probe_path("tensor")
    c.reset_stats()
    c.probe(Qd)
    # no more rechecked pairs than near-duplicates and a few close ones
    assert c.info()["candidates"] <= 300 * 40
    c.close()


@pytest.mark.parametrize("what", ["large", "small"])
def test_unfit_tables(dev, what):
    """Tables FP16 does not hold (overflow, the subnormal range) are screened in
    TF32, with the same results."""
    rng = np.random.default_rng(3)
    rows, Q = data(rng, 2000, 64, 300)
    s = np.float32(1e5 if what == "large" else 1e-6)
    rows, Q = rows * s, Q * s
    c = make(dev, 64, 5, rows)
    assert c.screen_info() == {"fp16": True, "fp16_copy": True, "unfit": 0}
    c.insert(torch.from_numpy(rows).to(dev))
    inf = c.screen_info()
    assert inf["fp16_copy"] and not inf["fp16"] and inf["unfit"] > c.size // 2
    same_as_exact(c, torch.from_numpy(Q).to(dev), ["tensor", "tensor_pair"])
    c.close()


@pytest.mark.parametrize("what", ["large", "small"])
@pytest.mark.parametrize("grow", ["insert", "unaligned", "scalar", "async", "select", "kcenter", "writeback"])
def test_unfit_entries_counted(dev, grow, what):
    """Every path that appends entries counts those whose FP16 copy does not
    serve: 3 among 500 whose copies do send the whole table to the TF32 screen,
    and queries next to them hit them. (The features of the small ones round to
    zero in FP16: an FP16 screen would lose their hits.) A table without such an
    entry stays in FP16."""
    d = 65 if grow == "scalar" else 64  # d % 4 != 0: features moved one by one
    rng = np.random.default_rng(11)
    rows, Q = data(rng, 500, d, 200)
    s = np.float32(1e5 if what == "large" else 1e-8)
    odd = rng.standard_normal((3, d)).astype(np.float32) * s
    near = odd[np.arange(30) % 3] + s * np.float32(1e-3) * rng.standard_normal((30, d)).astype(np.float32)

    def grown(rows):
        c = make(dev, d, 6, rows, capacity=1200)
        R = torch.from_numpy(rows).to(dev)
        if grow == "unaligned":
            buf = torch.zeros(rows.size + 1, device=dev)
            buf[1:] = R.reshape(-1)
            c.insert(buf[1:].view(rows.shape))
        elif grow == "async":
            for k in range(0, len(rows), 100):
                c.insert(R[k:k + 100], wait=False)
        elif grow in ("select", "kcenter"):
            c.insert_select(R, strategy="kcenter" if grow == "kcenter" else "radius_dedup",
                            budget_per_class=400 if grow == "kcenter" else 0)
        elif grow == "writeback":
            c.probe_writeback(R)
        else:
            c.insert(R)
        return c

    at = np.array([7, 250, 502])
    mixed = np.insert(rows, at - np.arange(3), odd, axis=0)
    assert np.array_equal(mixed[at], odd)
    c = grown(mixed)
    assert c.screen_info() == {"fp16": False, "fp16_copy": True, "unfit": 3}
    ref = same_as_exact(c, torch.from_numpy(np.concatenate([near, Q])).to(dev), ["tensor", "tensor_pair"])
    keys = c.entries()["keys"]
    assert (ref[0][:30] >= 0).all() and np.array_equal(keys[ref[0][:30]], odd[np.arange(30) % 3])
    c.close()
    c = grown(rows)
    assert c.screen_info() == {"fp16": True, "fp16_copy": True, "unfit": 0}
    c.close()


def test_extreme_queries(dev):
    """Queries of any magnitude are scaled into FP16's range by the prologue;
    NaN and infinite ones miss; a zero query gets the exact kernel's answer."""
    rng = np.random.default_rng(9)
    rows, Q = data(rng, 3000, 40, 400)
    for k, s in enumerate([1e30, 1e-30, 1e-38, 1e-42, 1e5, 1e-6, 0.0]):
        Q[k] *= np.float32(s)
    Q[10, 3], Q[11, 0], Q[12] = np.nan, np.inf, -np.inf
    Q[13, 1:] *= np.float32(1e-8)
    rows[0] = 0  # near the tiny queries
    c = make(dev, 40, 5, rows)
    c.insert(torch.from_numpy(rows).to(dev))
    ref = same_as_exact(c, torch.from_numpy(Q).to(dev), ["tensor", "tensor_pair"])
    assert np.all(ref[0][10:13] == -1)
    c.close()


@pytest.mark.parametrize("d,n,nq", [(64, 2000, 1), (20, 300, 65), (33, 5000, 2048), (33, 5000, 2049), (1000, 700, 30)])
def test_batches_in_a_row(dev, d, n, nq):
    """Batches of different sizes and paths follow one another on one handle
    (the exact kernel counts on the words the batch before left empty; kernels
    finalize batches of up to 2,048 themselves), an empty cache among them:
    each answers as a fresh cache does."""
    from paper_2608_13144_gb300.lipcache import LipCache
    rng = np.random.default_rng(d + nq)
    rows, Q = data(rng, n, d, nq)
    c = make(dev, d, 5, rows)
    Qd = torch.from_numpy(Q).to(dev)
    for path in ("exact", "auto"):  # empty cache: misses
        c.set_probe_path(path)
        assert (c.probe(Qd)[0].cpu().numpy() == -1).all()
    c.insert(torch.from_numpy(rows).to(dev))
    fresh = make(dev, d, 5, rows)
    fresh.insert(torch.from_numpy(rows).to(dev))
    fresh.set_probe_path("exact")
    ref = [t.cpu().numpy() for t in fresh.probe(Qd)]
    paths = ["exact", "auto"] + (["tensor", "tensor_pair"] if d <= 256 else [])
    for path in paths + paths[::-1]:
        c.set_probe_path(path)
        for k in (1, nq, max(1, nq // 2)):
            got = [t.cpu().numpy() for t in c.probe(Qd[:k])]
            for x, y in zip(ref, got):
                assert np.array_equal(x[:k].view(np.uint8), y.view(np.uint8)), (path, k)
    c.close()
    fresh.close()


@pytest.mark.parametrize("kind", ["fp16", "tf32"])
@pytest.mark.parametrize("radius", ["global", "coinciding"])
@pytest.mark.parametrize("B", [129, 257, 640])
def test_overflowing_radius_ragged_batch(dev, kind, radius, B):
    """Entries whose radius overflows have a screen term of -inf, which every
    query passes; the rows that fill the last query tile up must not: the
    screen rechecks no more than B x size pairs, and a larger exact batch
    afterwards finds no hit of theirs. The queries are the first rows of a
    larger buffer."""
    from paper_2608_13144_gb300.lipcache import LipCache
    n, d, C = 700, 48, 4
    rng = np.random.default_rng(B)
    s = np.float32(1.0 if kind == "fp16" else 1e5)  # 1e5: no FP16 copy of the keys serves
    rows = torch.from_numpy(rng.standard_normal((n, d)).astype(np.float32) * s).to(dev)
    buf = torch.from_numpy(rng.standard_normal((2048, d)).astype(np.float32) * s).to(dev)
    far = torch.from_numpy(rng.standard_normal((1024, d)).astype(np.float32) * s * np.float32(3)).to(dev)
    W = (rng.standard_normal((C, d)) / d).astype(np.float32) / s
    b = np.zeros(C, np.float32)
    if radius == "coinciding":  # every row the same: no class can take over, r* = +inf
        W[:] = W[0]
        b = np.arange(C, dtype=np.float32)

    def cache():
        c = LipCache(d, C, n, "tight", device=dev)
        c.set_head(torch.from_numpy(W).to(dev), torch.from_numpy(b).to(dev))
        c.insert(rows)
        c.set_probe_path("exact")
        return c

    c, fresh = cache(), cache()
    ref_far = [t.cpu().numpy() for t in fresh.probe(far)]
    if radius == "global":
        c.set_radius_policy("global", 1e30)
    ref = [t.cpu().numpy() for t in c.probe(buf[:B])]
    assert (ref[0] >= 0).all()
    for path in ("tensor", "tensor_single", "tensor_pair"):
        if radius == "global":
            c.set_radius_policy("global", 1e30)
        c.set_probe_path(path)
        c.reset_stats()
        got = [t.cpu().numpy() for t in c.probe(buf[:B])]
        for x, y in zip(ref, got):
            assert np.array_equal(x, y), path
        assert c.info()["candidates"] == B * c.size  # (every pair of a query passes, no other)
        if radius == "global":
            c.set_radius_policy("certified")
        c.set_probe_path("exact")
        for x, y in zip(ref_far, [t.cpu().numpy() for t in c.probe(far)]):
            assert np.array_equal(x, y), path
    c.close()
    fresh.close()


@pytest.mark.parametrize("B", [65535 * 64, 65535 * 64 + 1, 1 << 22])
def test_largest_exact_batches(dev, B):
    """The exact kernel on batches around the most query tiles a grid has rows
    for, up to the largest batch a probe takes."""
    rng = np.random.default_rng(5)
    rows = rng.standard_normal((70, 4)).astype(np.float32)
    c = make(dev, 4, 3, rows)
    c.insert(torch.from_numpy(rows).to(dev))
    c.set_probe_path("exact")
    R = torch.from_numpy(rows).to(dev)
    Q = R[torch.arange(B, device=dev) % 70]
    Q[1::2] += 1e3  # (misses)
    out = c.probe(Q)
    small = c.probe(Q[:140])
    for x, y in zip(small, out):
        want = x.repeat((B + 139) // 140)[:B]
        assert torch.equal(want, y)
    assert (small[0][::2] >= 0).any() and (small[0][1::2] == -1).all()
    c.close()
