"""The workloads by which this library's speed is judged: builds, batch
updates, k-NN, range queries and forests through the public Python binding,
from requests of a few dozen queries to 1e8 points.

Points are int32, uniform in [0, 2^30) or varden-like (a random walk with
rare restarts: dense clusters of about 1e4 points), as in the benchmark and
the tests.  They are drawn on the GPU from the seed alone.
"""
import math

import numpy as np
import torch

from paper_2411_09275_gb300 import pkd

LIMIT = 1 << 30
DEV = "cuda"
RESTART = 1e-4       # varden-like: probability of a restart per point
CLUSTER = 1 << 18    # varden-like: about how wide a cluster of 1 / RESTART points gets


def listed():
    base = {"points": "uniform", "phi": 32, "count_mode": 0, "given_ids": False}
    return [
        # One interactive request: a few dozen 10-NN queries on a resident 2-D
        # tree of 1e6 points.  Latency of one call.
        dict(base, name="knn_few", kind="knn", n=1_000_000, d=2, q=64, k=10, boxes=False, near=False),
        # A server's query batch: 10-NN of 1e5 positions taken from clustered 3-D
        # data (the upper end of the serving workload's query batches).
        dict(base, name="knn_serving", kind="knn", n=10_000_019, d=3, points="varden", q=100_000, k=10, boxes=False,
             near=True),
        # Bulk analysis: 10-NN of 1e6 independent positions, uniform 3-D data.
        dict(base, name="knn_bulk", kind="knn", n=10_000_000, d=3, q=1_000_000, k=10, boxes=False, near=False),
        # High dimension, many neighbours (feature vectors): k past the small-k
        # range, few subtrees can be pruned.
        dict(base, name="knn_wide", kind="knn", n=200_003, d=8, q=2_000, k=100, boxes=False, near=True),
        # The variant with stored bounding boxes, on clustered 5-D data.
        dict(base, name="knn_boxes", kind="knn", n=1_000_003, d=5, points="varden", q=20_000, k=10, boxes=True,
             near=True),
        # Window queries on clustered 2-D map data: how many points lie in each
        # of 1e4 windows, and which.
        dict(base, name="range", kind="range", n=3_000_017, d=2, points="varden", q=10_000, hits=300, boxes=False),
        # The smallest build in use: one tree of 2e4 points and a few queries.
        dict(base, name="build_small", kind="build", n=20_000, d=3, q=256, k=10),
        # 1e6 2-D points and 10-NN for 1e4 queries.
        dict(base, name="build_million", kind="build", n=1_000_000, d=2, q=10_000, k=10),
        # The benchmark's step: build 1e8 3-D uniform points, insert 1e7, delete
        # 1e7 of the stored ids.
        dict(base, name="step_uniform", kind="step", n=100_000_000, d=3, m=10_000_000, q=100_000, k=10),
        # The same step on clustered data at a tenth of the size, odd sizes,
        # ids given by the caller.
        dict(base, name="step_varden", kind="step", n=10_000_019, d=3, points="varden", m=1_000_003, q=10_000, k=10,
             given_ids=True),
        # A server's small update: 1e3 new points into a resident tree of 1e7,
        # a query batch that sees them, and their deletion.
        dict(base, name="update_small", kind="update", n=10_000_019, d=3, points="varden", m=1_000, q=1_000, k=10),
        # Many independent trees of uneven sizes in one call.
        dict(base, name="forest", kind="forest", trees=512, n=0, lo=1_000, hi=1_000_000, d=3, q=1_000, k=10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["knn", "knn", "knn", "range", "build", "step", "update", "forest"])
    d = rng.choice([1, 2, 2, 3, 3, 3, 4, 5, 6, 8])
    c = {"kind": kind, "d": d, "points": rng.choice(["uniform", "varden"]), "phi": rng.choice([32, 32, 32, 16]),
         "count_mode": rng.choice([0, 0, 0, 1]), "given_ids": rng.choice([False, True]), "k": 10}
    if d >= 5 and kind not in ("knn", "range"):
        c["points"] = "varden"
    # searches in many dimensions visit much of the tree: fewer points and queries there
    big = {1: 1.0, 2: 1.0, 3: 1.0, 4: 0.3, 5: 0.1}.get(d, 0.02)
    if kind == "knn":
        c["n"] = _log(rng, 10_000, max(200_000, 10_000_000 * big))
        c["k"] = rng.choice([1, rng.randint(2, 9), 10, 10, rng.randint(11, 16), rng.randint(17, 128)])
        c["q"] = _log(rng, 20, max(1_000, 1_000_000 * big * min(1.0, 16 / c["k"]) ** 1.5))
        if d >= 6:
            c["q"] = min(c["q"], 2_000)
        c["boxes"] = rng.random() < 0.2
        c["near"] = c["points"] == "varden" or rng.random() < 0.5
    elif kind == "range":
        c["n"] = _log(rng, 10_000, max(200_000, 10_000_000 * big))
        c["q"] = _log(rng, 20, 20_000 * max(big, 0.1))
        c["hits"] = _log(rng, 1, 1_000)
        c["boxes"] = rng.random() < 0.2
    elif kind == "build":
        c["n"] = _log(rng, 1_000, 20_000_000)
        c["q"] = _log(rng, 20, max(100, 10_000 * big))
    elif kind == "step":
        c["n"] = _log(rng, 100_000, 20_000_000)
        c["m"] = max(1, c["n"] // rng.randint(10, 100))
        c["q"] = _log(rng, 20, max(100, 10_000 * big))
    elif kind == "update":
        c["n"] = _log(rng, 1_000_000, 10_000_000)
        c["m"] = _log(rng, 100, c["n"] // 1_000)
        c["q"] = _log(rng, 20, max(100, 10_000 * big))
    else:
        c["trees"] = _log(rng, 4, 512)
        c["n"] = 0
        c["lo"] = _log(rng, 200, 2_000)
        c["hi"] = _log(rng, 10_000, 300_000)
        c["q"] = _log(rng, 20, max(100, 1_000 * big))
    return c


# --- inputs ------------------------------------------------------------------

def _points(kind, n, d, g):
    if kind == "uniform":
        return torch.randint(0, LIMIT, (n, d), generator=g, device=DEV, dtype=torch.int32)
    # varden-like: a random walk (steps uniform in [-L, L], L log-uniform in
    # [1, 1e4]), with restarts at uniform points, reflected into the domain
    step = torch.exp(torch.rand((n, 1), generator=g, device=DEV, dtype=torch.float64) * math.log(1e4))
    step = ((torch.rand((n, d), generator=g, device=DEV, dtype=torch.float64) * 2 - 1) * step).round_().to(torch.int64)
    new = torch.rand(n, generator=g, device=DEV) < RESTART
    new[0] = True
    at = torch.nonzero(new).reshape(-1)
    seg = torch.cumsum(new, 0) - 1
    start = torch.randint(0, LIMIT, (at.numel(), d), generator=g, device=DEV, dtype=torch.int64)
    walk = torch.cumsum(step, 0)
    x = walk.add_((start - walk[at])[seg]).remainder_(2 * LIMIT)
    return torch.where(x >= LIMIT, 2 * LIMIT - 1 - x, x).to(torch.int32).contiguous()


def _sizes(case, seed):
    r = np.random.default_rng(seed)
    s = np.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"]), case["trees"])).astype(np.int64)
    return np.concatenate([[0], np.cumsum(s)])


def _params(case):
    return pkd.Params(d=case["d"], phi=case["phi"], count_mode=case["count_mode"])


def _inputs(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    d, kind = case["d"], case["kind"]
    s = {"case": case}
    if kind == "forest":
        s["offsets"] = _sizes(case, seed)
    n = int(s["offsets"][-1]) if kind == "forest" else case["n"]
    m = case.get("m", 0)
    s["x"] = _points(case["points"], n, d, g)
    # ids: positions, or labels of the caller's own
    s["ids"] = torch.arange(n + m, device=DEV, dtype=torch.int32)
    if case["given_ids"]:
        s["ids"] = torch.randperm(n + m, generator=g, device=DEV).to(torch.int32)
    if m:
        # new points of the same distribution (a walk of their own); a server's
        # small batch also has points all over the stored ones
        s["new"] = _points(case["points"], m, d, g)
        if kind == "update":
            half = m // 2
            at = torch.randint(0, n, (half,), generator=g, device=DEV)
            move = torch.randint(-1000, 1001, (half, d), generator=g, device=DEV, dtype=torch.int32)
            s["new"][:half] = (s["x"][at] + move).clamp_(0, LIMIT - 1)
        s["new_ids"] = s["ids"][n:].contiguous()
        s["ids"] = s["ids"][:n].contiguous()
    if kind == "step":
        s["gone"] = s["ids"][torch.randperm(n, generator=g, device=DEV)[:m]].contiguous()
    q = case["q"]
    if kind == "range":
        hits = min(case["hits"], 3_000)
        side = LIMIT * min(1.0, hits / n) ** (1 / d)
        if case["points"] == "varden":
            side = CLUSTER * min(1.0, hits * RESTART) ** (1 / d)
        half = side / 2 * torch.exp2(torch.rand((q, d), generator=g, device=DEV, dtype=torch.float64) - 0.5)
        mid = s["x"][torch.randint(0, n, (q,), generator=g, device=DEV)].double()
        s["lo"] = (mid - half).clamp_(0, LIMIT - 1).to(torch.int32).contiguous()
        s["hi"] = (mid + half).clamp_(0, LIMIT - 1).to(torch.int32).contiguous()
        return s
    if kind == "forest":  # queries on some of the trees, each at that tree's points
        s["queries"] = [(t, _queries(case, s["x"][s["offsets"][t]:s["offsets"][t + 1]], g)) for t in _asked(case)]
    else:
        s["q"] = _queries(case, s["x"], g)
    return s


def _asked(case):
    return range(0, case["trees"], max(1, case["trees"] // 8))


def _queries(case, x, g):
    q, d = case["q"], case["d"]
    if not case.get("near", case["points"] == "varden"):
        return torch.randint(0, LIMIT, (q, d), generator=g, device=DEV, dtype=torch.int32)
    at = torch.randint(0, x.shape[0], (q,), generator=g, device=DEV)  # stored positions, moved a little
    move = torch.randint(-1000, 1001, (q, d), generator=g, device=DEV, dtype=torch.int32)
    return (x[at] + move).clamp_(0, LIMIT - 1).contiguous()


def prepare(case, seed):
    s = _inputs(case, seed)
    if case["kind"] in ("knn", "range", "update"):  # the resident tree
        s["tree"] = pkd.Tree(s["x"], s["ids"] if case["given_ids"] else None, _params(case))
        if case.get("boxes"):
            pkd.pkd_set_bounding_boxes(s["tree"]._h, True)
    return s


# --- one pass ----------------------------------------------------------------

def run(s):
    case = s["case"]
    kind, k = case["kind"], case.get("k")
    ids = s["ids"] if case["given_ids"] else None
    if kind == "knn":
        return s["tree"].knn(s["q"], k)
    if kind == "range":
        # the counts, and the points of every window: those of any window are marked
        t = s["tree"]
        counts = t.range_count(s["lo"], s["hi"])
        offsets, found = pkd.pkd_range_report(t._h, s["lo"], s["hi"])
        marked = torch.zeros(case["n"], dtype=torch.bool, device=DEV)
        marked.index_fill_(0, found.long(), True)
        return {"counts": counts, "offsets": offsets, "marked": marked}
    if kind == "build":
        t = pkd.Tree(s["x"], ids, _params(case))
        out = t.knn(s["q"], k)
        t.close()
        return out
    if kind == "step":
        t = pkd.Tree(s["x"], ids, _params(case))
        t.insert(s["new"], s["new_ids"])
        gone = t.delete(s["gone"])
        out_i, out_d = t.knn(s["q"], k)
        size = t.size
        t.close()
        return {"ids": out_i, "d2": out_d, "deleted": gone, "size": size}
    if kind == "update":
        t = s["tree"]
        t.insert(s["new"], s["new_ids"])
        out_i, out_d = t.knn(s["q"], k)
        return {"ids": out_i, "d2": out_d, "deleted": t.delete(s["new_ids"]), "size": t.size}
    f = pkd.pkd_build_forest(s["x"], ids, s["offsets"], _params(case))
    out = []
    for tree, queries in s["queries"]:
        oi = torch.empty((case["q"], k), dtype=torch.int32, device=DEV)
        od = torch.empty((case["q"], k), dtype=torch.int64, device=DEV)
        pkd.pkd_forest_knn(f, tree, queries, k, oi, od)
        out += [oi, od]
    pkd.pkd_forest_free(f)
    return out


# --- what a pass cannot do without --------------------------------------------

def work(case):
    d, kind, q, k = case["d"], case["kind"], case["q"], case.get("k", 10)
    point = 4 * d + 4
    # a search reads its query and at least the points that it returns
    per_query, per_query_ops = 4 * d + k * (point + 12), 3 * d * k
    if kind == "knn":
        return {"bytes": q * per_query, "flops": q * per_query_ops}
    if kind == "range":
        hits = min(case["hits"], 3_000, case["n"])
        return {"bytes": q * (16 * d + 24 + hits * (2 * 4 * d + 8)) + case["n"], "flops": 4 * q * hits * d}
    if kind == "update":
        m = case["m"]
        return {"bytes": 2 * m * point + 4 * m + q * per_query, "flops": q * per_query_ops}
    # a build reads every point and writes it and its id into its leaf
    n, runs = case["n"], 1
    if kind == "forest":
        n = case["trees"] * (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        runs = len(_asked(case))
    b = n * (4 * d + (4 if case["given_ids"] else 0) + point) + runs * q * per_query
    if kind == "step":
        b += 2 * case["m"] * point + 4 * case["m"]
    return {"bytes": b, "flops": runs * q * per_query_ops}


def exact(case, seed):
    """Distances and counts by brute force in 64 bits (ids, which ties decide,
    and trees too large for it are left out)."""
    if case["kind"] not in ("knn", "range", "build") or case["n"] * case["q"] * case["d"] > 1e11:
        return None
    s = _inputs(case, seed)
    x, n, q, d = s["x"].to(torch.int64), case["n"], case["q"], case["d"]
    rows = max(1, 50_000_000 // n)
    out = []
    for a in range(0, q, rows):
        b = min(q, a + rows)
        if case["kind"] == "range":
            inside = torch.ones((b - a, n), dtype=torch.bool, device=DEV)
            for j in range(d):
                inside &= (x[None, :, j] >= s["lo"][a:b, j, None]) & (x[None, :, j] <= s["hi"][a:b, j, None])
            out.append(inside.sum(1))
        else:
            d2 = torch.zeros((b - a, n), dtype=torch.int64, device=DEV)
            for j in range(d):
                d2 += (x[None, :, j] - s["q"][a:b, j, None].to(torch.int64)) ** 2
            out.append(torch.topk(d2, case["k"], dim=1, largest=False, sorted=True).values)
    got = torch.cat(out)
    return {"counts": got, "offsets": None, "marked": None} if case["kind"] == "range" else (None, got)
