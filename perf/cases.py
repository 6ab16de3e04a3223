"""Timed cases of the certified cache lookup, through the public binding.

Five kinds of pass, each what a program using the cache runs:

* probe:  one lookup of a query batch in a cache built beforehand (Algorithm 2), the call a serving loop repeats;
* build:  Algorithm 1 from nothing: create the cache, install the head (its spectral norm), certify and insert every
          row in batches, answer a first query batch, drop the cache;
* select: the same with the default selection strategy of Sec. 5.5 and a per-class budget;
* serve:  a session with write-back: a small cache is seeded, then query batches are looked up and their certified
          misses appended (Algorithm 2 with its write-back flag);
* audit:  a lookup followed by the certified-consistency check of its hits (reported with every experiment of Sec. 5).

Features are Gaussian mixtures in the feature space (one component per class; centre norm and spread grow with d as in
synth.py's workloads), heads are Gaussian, optionally rescaled to unit spectral norm (Lipschitz-constrained), and a
share of the queries are near-duplicates of cached rows.
"""
import math

import numpy as np
import torch

from paper_2608_13144_gb300.lipcache import LipCache

DEV = torch.device("cuda", 0)
FIRST_QUERIES = 256  # queries answered by a freshly built cache


def listed():
    def probe(name, d, classes, entries, batch, dup, noise, unit, radius="conservative"):
        return {"name": name, "kind": "probe", "d": d, "classes": classes, "entries": entries, "batch": batch,
                "dup": dup, "noise": noise, "unit": unit, "radius": radius}

    return [
        # One query at a time against the paper's edge cache (200 entries per class, 10 classes, d = 64): pure latency.
        probe("probe_single", 64, 10, 2000, 1, 0.5, 0.02, False, "tight"),
        # CIFAR-10-shaped serving batch.
        probe("probe_cifar10", 64, 10, 50_000, 256, 0.4, 0.02, False),
        # CIFAR-100-shaped serving batch.
        probe("probe_cifar100", 128, 100, 50_000, 1024, 0.3, 0.01, False),
        # Tiny-ImageNet-shaped offline evaluation batch.
        probe("probe_tinyimagenet", 256, 200, 100_000, 4096, 0.3, 0.002, True),
        # Scale: the 4M-entry cache, 4,096 queries.
        probe("probe_scale", 128, 200, 4_000_000, 4096, 0.35, 0.002, True),
        # Wide features (the width of a small residual network's last layer, odd on purpose) and ragged sizes.
        probe("probe_wide_odd", 500, 100, 49_999, 1001, 0.3, 0.01, False),
        # The paper's edge cache built with its default (tight) radius: latency of head and small insert.
        {"name": "build_edge", "kind": "build", "d": 64, "classes": 10, "rows": 2000, "insert_batch": 2000,
         "dup": 0.4, "noise": 0.02, "unit": False, "radius": "tight"},
        # Tiny-ImageNet-shaped cache, tight radius, two insert calls (the second one ragged).
        {"name": "build_tinyimagenet", "kind": "build", "d": 256, "classes": 200, "rows": 100_000,
         "insert_batch": 65_536, "dup": 0.3, "noise": 0.002, "unit": True, "radius": "tight"},
        # Bulk build at the scale workload's shape, conservative radius, asynchronous inserts of 65,536 rows.
        {"name": "build_bulk", "kind": "build", "d": 128, "classes": 200, "rows": 1_900_000, "insert_batch": 65_536,
         "dup": 0.25, "noise": 0.002, "unit": True, "radius": "conservative"},
        # The paper's construction: radius-prioritised de-duplication of a CIFAR-10-sized pool, 200 entries per class.
        {"name": "select_cifar10", "kind": "select", "d": 64, "classes": 10, "rows": 50_000, "per_class": 200,
         "dup": 0.3, "noise": 0.02, "unit": False, "radius": "tight"},
        # A serving session that grows its cache: 12 batches of 250 queries (uneven) on 2,000 seeded entries.
        {"name": "serve_writeback", "kind": "serve", "d": 64, "classes": 10, "rows": 2000, "batch": 250, "batches": 12,
         "dup": 0.4, "noise": 0.02, "unit": False, "radius": "tight"},
        # Evaluation of a 10,000-query test set: lookup and consistency of the hits.
        {"name": "audit_cifar100", "kind": "audit", "d": 128, "classes": 100, "entries": 50_000, "batch": 10_000,
         "dup": 0.3, "noise": 0.01, "unit": False, "radius": "conservative"},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choices(["probe", "build", "select", "serve", "audit"], [10, 5, 2, 2, 2])[0]
    c = {"kind": kind, "d": log(12, 512 if kind == "probe" else 256), "classes": log(3, 200),
         "dup": round(rng.uniform(0.1, 0.5), 2), "noise": rng.choice([0.002, 0.01, 0.02, 0.05]),
         "unit": rng.random() < 0.5, "radius": rng.choice(["conservative", "tight"])}
    if rng.random() < 0.4:
        c["d"] = max(16, c["d"] // 16 * 16)
    if kind == "probe":
        c["batch"] = log(1, 4096)
        most = 2_000_000_000_000 if c["d"] <= 256 else 200_000_000_000
        c["entries"] = max(300, min(log(300, 4_000_000), most // (c["batch"] * c["d"]), 500_000_000 // c["d"]))
    elif kind == "audit":
        c["entries"], c["batch"] = log(1000, 100_000), log(50, 10_000)
    elif kind == "serve":
        c["rows"], c["batch"], c["batches"] = log(500, 20_000), log(1, 1024), rng.randint(2, 12)
    elif kind == "select":
        c["rows"], c["per_class"] = log(2000, 50_000), log(20, 300)
    else:
        most = 20_000_000_000 if c["radius"] == "conservative" else 5_000_000_000
        c["rows"] = max(300, min(log(500, 1_000_000), most // (c["classes"] * c["d"])))
        c["insert_batch"] = max(log(256, 65_536), -(-c["rows"] // 24))
    return c


# ---------------------------------------------------------------- inputs
class State:
    pass


def _mixture(gen, centres, n, spread):
    x = torch.randn(n, centres.shape[1], generator=gen, device=DEV)
    pick = torch.randint(0, centres.shape[0], (n,), generator=gen, device=DEV)
    return x.mul_(spread).add_(centres[pick])


def _inputs(case, seed):
    """(W, b, rows, queries) of a case, on the GPU."""
    d, classes = case["d"], case["classes"]
    host = np.random.default_rng([seed, 17])
    W = host.standard_normal((classes, d)) / math.sqrt(d)
    if case["unit"]:
        W = W / np.linalg.norm(W, 2)
    b = host.standard_normal(classes) * 0.1
    ctr = host.standard_normal((classes, d))
    ctr *= 4.0 * (d / 16.0) ** 0.33 / np.linalg.norm(ctr, axis=1, keepdims=True)
    W, b, ctr = (torch.from_numpy(x.astype(np.float32)).to(DEV) for x in (W, b, ctr))
    spread = 0.5 * (d / 16.0) ** 0.17
    gen = torch.Generator(device=DEV).manual_seed(seed * 1_000_003 + 7)
    n = case["entries"] if "entries" in case else case["rows"]
    rows = _mixture(gen, ctr, n, spread)
    if case["kind"] == "select":
        # a pool with repeats: every third row is a near-duplicate of the row before it
        rows[1::3] = rows[0::3][:rows[1::3].shape[0]] + case["noise"] * torch.randn(
            rows[1::3].shape, generator=gen, device=DEV)
    nq = {"probe": case.get("batch"), "audit": case.get("batch"),
          "serve": case.get("batch", 0) * case.get("batches", 0)}.get(case["kind"], FIRST_QUERIES)
    Q = _mixture(gen, ctr, nq, spread)
    near = torch.rand(nq, generator=gen, device=DEV) < case["dup"]
    src = torch.randint(0, n, (nq,), generator=gen, device=DEV)
    jitter = torch.randn(nq, d, generator=gen, device=DEV) * case["noise"]
    Q = torch.where(near[:, None], rows[src] + jitter, Q).contiguous()
    return W, b, rows, Q


def prepare(case, seed):
    s = State()
    s.case = case
    s.W, s.b, rows, Q = _inputs(case, seed)
    if case["kind"] in ("probe", "audit"):
        s.cache = LipCache(case["d"], case["classes"], case["entries"], case["radius"], device=DEV)
        s.cache.set_head(s.W, s.b)
        for k in range(0, rows.shape[0], 65_536):
            s.cache.insert(rows[k:k + 65_536])
        s.cache.reserve(case["batch"])
        s.Q = Q
    elif case["kind"] == "serve":
        s.rows, s.Q = rows, list(Q.split(case["batch"]))
    else:
        s.rows, s.Q = rows, Q
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    case = s.case
    if case["kind"] == "probe":
        return s.cache.probe(s.Q)
    if case["kind"] == "audit":
        index, label, dist = s.cache.probe(s.Q)
        consistent, n_hits, n_consistent = s.cache.consistency(s.Q, index)
        return index, label, dist, consistent, n_hits, n_consistent
    n = s.rows.shape[0]
    # (selection wants room for every candidate its budgets might admit)
    capacity = n + sum(q.shape[0] for q in s.Q) if case["kind"] == "serve" else n
    out = {"inserted": []}
    with LipCache(case["d"], case["classes"], capacity, case["radius"], device=DEV) as cache:
        out["sigma"] = cache.set_head(s.W, s.b)
        if case["kind"] == "build":
            for k in range(0, n, case["insert_batch"]):
                index, radius, _ = cache.insert(s.rows[k:k + case["insert_batch"]], wait=False)
                out["inserted"].append((index, radius))
            out["first"] = cache.probe(s.Q)
            out["size"] = cache.size
        elif case["kind"] == "select":
            out["inserted"] = cache.insert_select(s.rows, strategy="radius_dedup", budget_per_class=case["per_class"])
            out["first"] = cache.probe(s.Q)
        else:
            out["inserted"] = cache.insert(s.rows)
            out["served"] = [cache.probe_writeback(q) for q in s.Q]
    return out


# ---------------------------------------------------------------- accounting
def _probe_work(n, d, q):
    return n * (4 * d + 4) + q * (4 * d + 16), 2 * n * d * q


def _certify_work(n, d, classes):
    # rows read, keys and six fields written, index and radius written
    return n * (8 * d + 24 + 12), 2 * n * d * classes


def work(case):
    d, classes = case["d"], case["classes"]
    total = [4 * d * classes, 0]

    def add(w, times=1):
        total[0] += w[0] * times
        total[1] += w[1] * times

    if case["kind"] in ("probe", "audit"):
        add(_probe_work(case["entries"], d, case["batch"]))
        if case["kind"] == "audit":
            add((case["batch"] * (4 * d + 9), 2 * case["batch"] * d * classes))
    elif case["kind"] == "serve":
        add(_certify_work(case["rows"], d, classes))
        for k in range(case["batches"]):
            add(_probe_work(case["rows"] + k * case["batch"] // 2, d, case["batch"]))
            add(_certify_work(case["batch"], d, classes))
    else:
        add(_certify_work(case["rows"], d, classes))
        kept = case["rows"] if case["kind"] == "build" else min(case["rows"], case["per_class"] * classes)
        add(_probe_work(kept, d, FIRST_QUERIES))
        if case["kind"] == "select":
            add((0, case["rows"] * kept * d))  # every candidate against the entries kept before it
    return {"bytes": total[0], "flops": total[1]}


def tolerance(case):
    # Distances are FP32 sums and radii FP32 roundings of nearly exact values: within 6e-8 of the 64-bit values in
    # 2-norm on every case (measured); no single radius may be off by more than 1e-5. Decisions, indices and labels
    # are whole values.
    t = {"rel": 3e-7, "max": 1e-5, "differ": 0.0}
    if case["kind"] == "select":
        t["differ"] = 2e-3  # a candidate within rounding of a ball's edge changes the greedy selection after it
    return t


# ---------------------------------------------------------------- 64-bit values
def _radii64(case, W, b, rows):
    """(radius, label) of every row: Eq. 21 or Eq. 29 in 64 bits."""
    W, b = W.double(), b.double()
    sigma = float(np.linalg.norm(W.cpu().numpy(), 2))
    pair = torch.cdist(W, W, compute_mode="donot_use_mm_for_euclid_dist")
    radius, label = [], []
    for z in rows.split(65_536):
        s = z.double() @ W.T + b
        top, at = s.topk(2, dim=1)
        if case["radius"] == "conservative":
            r = (top[:, 0] - top[:, 1]) / (sigma * math.sqrt(2.0))
        else:
            t = (top[:, :1] - s) / pair[at[:, 0]]
            t.scatter_(1, at[:, :1], math.inf)
            r = t.min(dim=1).values
        radius.append(r)
        label.append(at[:, 0].int())
    return sigma, torch.cat(radius), torch.cat(label)


def _probe64(keys, radius, label, Q):
    """Nearest entry strictly inside its ball, by brute force in 64 bits."""
    q = Q.double()
    qn = (q * q).sum(1)
    best = torch.full((q.shape[0],), math.inf, dtype=torch.float64, device=DEV)
    index = torch.full((q.shape[0],), -1, dtype=torch.int64, device=DEV)
    first = 0
    for k, r in zip(keys.split(32_768), radius.split(32_768)):
        k = k.double()
        d2 = torch.addmm(qn[:, None] + (k * k).sum(1)[None, :], q, k.T, alpha=-2.0).clamp_(min=0.0)
        d2.masked_fill_(d2 >= (r * r)[None, :], math.inf)
        m, at = d2.min(dim=1)
        near = m < best
        best = torch.where(near, m, best)
        index = torch.where(near, at + first, index)
        first += k.shape[0]
    hit = index >= 0
    at = index.clamp(min=0)
    dist = torch.where(hit, (q - keys[at].double()).norm(dim=1), math.inf)
    return index, torch.where(hit, label[at], -1), dist


def exact(case, seed):
    W, b, rows, Q = _inputs(case, seed)
    sigma, radius, label = _radii64(case, W, b, rows)
    keep = radius > 0
    index = torch.where(keep, torch.cumsum(keep, 0) - 1, -1)
    if case["kind"] == "select":
        return {"inserted": (None, radius, None), "sigma": sigma, "first": (None, None, None)}
    keys, kr, kl = rows[keep], radius[keep], label[keep]
    if case["kind"] == "serve":
        served = []
        for q in Q.split(case["batch"]):
            i, lab, dist = _probe64(keys, kr, kl, q)
            _, r, y = _radii64(case, W, b, q)
            new = (i < 0) & (r > 0)
            ins = torch.where(new, torch.cumsum(new, 0) - 1 + keys.shape[0], -1)
            served.append((i, lab, dist, ins, int(new.sum())))
            keys, kr, kl = torch.cat([keys, q[new]]), torch.cat([kr, r[new]]), torch.cat([kl, y[new]])
        return {"inserted": (index, radius, int(keep.sum())), "sigma": sigma, "served": served}
    found = _probe64(keys, kr, kl, Q)
    if case["kind"] == "probe":
        return found
    if case["kind"] == "audit":
        hit = found[0] >= 0
        same = (_radii64(case, W, b, Q)[2] == kl[found[0].clamp(min=0)]) & hit
        return (*found, torch.where(hit, same.to(torch.int8), -1), int(hit.sum()), int(same.sum()))
    batch = case["insert_batch"]
    return {"inserted": list(zip(index.split(batch), radius.split(batch))), "sigma": sigma, "first": found,
            "size": int(keep.sum())}
