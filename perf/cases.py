"""Timed cases over the library's public Python interface.

A case is one kind of call sequence at one size:

query    k-NN of one query batch on a resident forest (Forest.knn)
plan     the same through a prepared k-NN plan (KnnPlan.launch), as in a serving loop
step     a batch of points inserted, a batch of live ids erased, then k-NN, on a resident forest
build    a forest made from its points, asked once and closed (a structure rebuilt per frame)
forests  one step on many independent forests, one batched call per operation

The request server is left out: it issues these same calls from threads of its own, and how
requests are grouped there depends on the host's scheduling from pass to pass.

Every result is an integer (ids and exact squared distances), so every case is "exact".
"""
import math
import random

import torch

from paper_2112_06188_gb300.forest import Forest, KnnPlan, erase_batch, insert_batch, knn_batch

GRID = 1 << 20          # coordinates lie in [0, 2^20)
ROUNDS = 16             # insert batches and erase sets that a step case goes through in turn
EXACT_PAIRS = 2e10      # most point-query pairs that exact() goes through

_BASE = {"data": "uniform", "leaf": 16, "split": "object", "forests": 1, "batch": 0, "near": True}


def _case(name, kind, **kw):
    c = dict(_BASE, kind=kind)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a lone question to a small map: nothing but latency
        _case("query_2d_one", "query", dim=2, n=65_536, queries=1, k=5, near=False),
        # a serving request of ordinary size (1 to 100,000 queries, log-uniform: a few hundred)
        _case("query_5d_316", "query", dim=5, n=1_000_000, queries=316, k=10, near=False),
        # nearest neighbours for a million points of a large scan
        _case("query_3d_1m", "query", dim=3, n=10_000_000, queries=1_000_000, k=10),
        # feature vectors of varying density, the largest case
        _case("query_7d_clusters", "query", dim=7, n=10_000_000, queries=1_000_000, k=5, data="clusters"),
        # a wide neighbourhood in a dimension without a kernel of its own, other leaves
        _case("query_4d_k32", "query", dim=4, n=500_003, queries=100_003, k=32, leaf=24),
        # the highest dimension, small requests through a prepared plan
        _case("plan_16d", "plan", dim=16, n=50_000, queries=1_000, k=8, data="clusters"),
        # the small workload: a batch in, a batch out, a batch of questions
        _case("step_2d_small", "step", dim=2, n=65_536, batch=8_192, queries=4_096, k=5, near=False),
        # serving-sized updates
        _case("step_5d_10k", "step", dim=5, n=1_000_000, batch=10_007, queries=1_009, k=5, near=False),
        # the headline step
        _case("step_3d_10m", "step", dim=3, n=10_000_000, batch=1_000_000, queries=1_000_000, k=10),
        # the splitting rule of moving, clustered 2-D data
        _case("step_2d_spatial", "step", dim=2, n=1_000_000, batch=100_000, queries=100_000, k=5,
              data="clusters", split="spatial"),
        # a large static build, asked once
        _case("build_3d_10m", "build", dim=3, n=10_000_000, queries=4_096, k=10),
        # hundreds of independent maps in shared launches; n is the largest map
        _case("forests_512", "forests", dim=3, forests=512, n=200_000, batch=10, queries=3_000, k=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["query", "query", "plan", "step", "step", "build", "forests"])
    if kind == "forests":
        return _case(None, kind, dim=rng.choice([2, 3]), forests=_log_int(rng, 3, 512), n=_log_int(rng, 2_000, 200_000),
                     batch=rng.randint(4, 20), queries=_log_int(rng, 50, 3_000), k=rng.choice([1, 5, 8, 10]))
    dim = rng.choice([2, 2, 3, 3, 3, 4, 5, 6, 7, 10, 16, rng.randint(1, 16)])
    top_n = 10_000_000 if dim <= 3 else 4_000_000 if dim <= 5 else 1_000_000 if dim <= 7 else 50_000
    top_m = 1_000_000 if dim <= 3 else 200_000 if dim <= 5 else 50_000 if dim <= 7 else 1_000
    data = rng.choice(["uniform", "clusters"]) if dim <= 7 else "clusters"
    n = _log_int(rng, 2_000, top_n)
    c = _case(None, kind, dim=dim, n=n, queries=_log_int(rng, 1, top_m), k=rng.choice([1, 2, 5, 8, 10, 16, 32]), data=data,
              leaf=rng.choice([8, 16, 16, 24, 32]), near=rng.random() < 0.5, split=rng.choice(["object"] * 4 + ["spatial"]))
    if kind == "step":
        c["batch"] = _log_int(rng, max(1, n // 1000), max(2, n // 8))
    if kind == "build":
        c["queries"] = min(c["queries"], 4_096)
    return c


# ---- inputs ----------------------------------------------------------------

class _Source:
    """Points of one distribution, drawn on the GPU from one seed."""

    def __init__(self, data, dim, seed):
        self.data, self.dim = data, dim
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)
        if data == "clusters":      # 100 Gaussian clusters, widths log-uniform in [2^8, 2^16]
            self.centre = torch.rand(100, dim, generator=self.g, device="cuda") * GRID
            self.sigma = torch.exp2(8 + 8 * torch.rand(100, generator=self.g, device="cuda"))

    def ints(self, hi, size):
        return torch.randint(0, hi, size, generator=self.g, device="cuda", dtype=torch.int64)

    def points(self, n):
        if self.data == "uniform":
            return torch.randint(0, GRID, (n, self.dim), generator=self.g, device="cuda", dtype=torch.int32)
        w = self.ints(100, (n,))
        x = torch.randn(n, self.dim, generator=self.g, device="cuda").mul_(self.sigma[w].unsqueeze(1)).add_(self.centre[w])
        return x.round_().clamp_(0, GRID - 1).to(torch.int32)

    def positions(self, n, count):
        """`count` distinct positions below n."""
        return torch.randperm(n, generator=self.g, device="cuda")[:count].clone()


def _fresh(batch, step):
    """The batch's points in pass `step`: the low bits differ each time, so that no point comes twice."""
    return torch.bitwise_xor(batch, step & 255)


class _World:
    """The inputs of a case on one forest, and the live set after the updates so far."""

    def __init__(self, case, seed):
        dim, n = case["dim"], case["n"]
        src = _Source(case["data"], dim, seed)
        self.points = src.points(n)
        # an update before the questions leaves a resident forest with several trees,
        # a part-filled buffer, tombstones and bloom filters
        churn = max(1, n // 20) if case["kind"] in ("query", "plan", "step") else 0
        self.churn = [(src.points(churn), src.positions(n, churn)) for _ in range(3 if churn else 0)]
        b = case["batch"]
        rounds = ROUNDS if case["kind"] == "step" else 0
        self.batches = [src.points(b) for _ in range(rounds)]
        self.out = [src.positions(n, b) for _ in range(rounds)]
        m = case["queries"]
        self.queries = self.points[src.ints(n, (m,))].contiguous() if case["near"] else src.points(m)


def _resident(case, w):
    """The forest after the first updates, and the ids it holds."""
    f = Forest(case["dim"], leaf_size=case["leaf"], split=case["split"])
    live = f.insert(w.points)
    for pts, gone in w.churn:
        new = f.insert(pts)
        f.erase(live[gone])
        live[gone] = new
    return f, live


def _forest_sizes(case):
    """Sizes log-uniform in [n / 200, n], each forest's batch and query count."""
    r = random.Random(case["n"])
    lo = max(100, case["n"] // 200)
    n = [_log_int(r, lo, case["n"]) for _ in range(case["forests"])]
    b = [max(1, x * case["batch"] // 100) for x in n]
    m = [r.randint(max(1, case["queries"] // 3), case["queries"] * 5 // 3) for _ in n]
    return n, b, m


class _Many:
    """The inputs of a case on many forests, laid out one forest after another."""

    def __init__(self, case, seed):
        self.n, self.b, self.m = _forest_sizes(case)
        src = _Source(case["data"], case["dim"], seed)
        self.points = src.points(sum(self.n)).split(self.n)
        self.batches = [src.points(sum(self.b)) for _ in range(ROUNDS)]
        # distinct positions of each forest: a stride through it from a random start
        first = torch.tensor([0] + self.n[:-1], device="cuda").cumsum(0)
        size, count = torch.tensor(self.n, device="cuda"), torch.tensor(self.b, device="cuda")
        rank = torch.arange(sum(self.b), device="cuda") - (count.cumsum(0) - count).repeat_interleave(count)
        stride = (size // count).repeat_interleave(count)
        size_r, first_r = size.repeat_interleave(count), first.repeat_interleave(count)
        self.out = [first_r + (rank * stride + src.ints(1 << 30, (len(self.n),)).repeat_interleave(count)) % size_r
                    for _ in range(ROUNDS)]
        self.queries = [p[src.ints(p.shape[0], (m,))].contiguous() for p, m in zip(self.points, self.m)]


def prepare(case, seed):
    k, dim, kind = case["k"], case["dim"], case["kind"]
    s = {"case": case, "pass": 0}
    if kind == "forests":
        w = _Many(case, seed)
        s["forests"] = [Forest(dim, leaf_size=case["leaf"]) for _ in w.n]
        ids = insert_batch(s["forests"], w.points)
        s["live"] = torch.cat(ids)
        m = sum(w.m)
        s["oi"] = torch.empty((m, k), dtype=torch.int32, device="cuda")
        s["od"] = torch.empty((m, k), dtype=torch.int64, device="cuda")
        s["rows"] = list(zip(s["oi"].split(w.m), s["od"].split(w.m)))
        s["world"] = w
        return s
    w = _World(case, seed)
    s["world"] = w
    if kind == "build":
        return s
    s["forest"], s["live"] = _resident(case, w)
    m = case["queries"]
    s["out"] = (torch.empty((m, k), dtype=torch.int32, device="cuda"), torch.empty((m, k), dtype=torch.int64, device="cuda"))
    if kind == "plan":
        s["plan"] = KnnPlan([s["forest"]], [w.queries], k, out=[s["out"]])
    return s


def run(state):
    case, w = state["case"], state["world"]
    kind, k = case["kind"], case["k"]
    if kind == "query":
        ids, d2 = state["forest"].knn(w.queries, k, out=state["out"])
        return {"ids": ids, "d2": d2}
    if kind == "plan":
        (ids, d2), = state["plan"].launch()
        return {"ids": ids, "d2": d2}
    if kind == "build":
        f = Forest(case["dim"], leaf_size=case["leaf"], split=case["split"])
        new = f.insert(w.points)
        ids, d2 = f.knn(w.queries, k)
        f.close()
        return {"new": new, "ids": ids, "d2": d2}
    at = state["pass"]
    state["pass"] = at + 1
    pts, gone = _fresh(w.batches[at % ROUNDS], at), w.out[at % ROUNDS]
    if kind == "step":
        new = state["forest"].insert(pts)
        count = state["forest"].erase(state["live"][gone])
        state["live"][gone] = new
        ids, d2 = state["forest"].knn(w.queries, k, out=state["out"])
        return {"new": new, "erased": count, "ids": ids, "d2": d2}
    new = torch.cat(insert_batch(state["forests"], pts.split(w.b)))
    counts = erase_batch(state["forests"], state["live"][gone].split(w.b))
    state["live"][gone] = new
    knn_batch(state["forests"], w.queries, k, out=state["rows"])
    return {"new": new, "erased": torch.tensor(counts), "ids": state["oi"], "d2": state["od"]}


# ---- what a pass needs, and what it has to give ------------------------------

def work(case):
    """Each input read once and each output written once; for k-NN also the k neighbours' coordinates."""
    d, k = case["dim"], case["k"]
    if case["kind"] == "forests":
        n, b, m = (sum(x) for x in _forest_sizes(case))
    else:
        n, b, m = case["n"], case["batch"], case["queries"]
    row = 4 * d + 12 * k                       # a query in, its ids and distances out
    by = m * (row + 4 * d * k)
    fl = m * k * 3.0 * d                       # the squared distances that are returned
    if case["kind"] in ("step", "forests"):
        by += b * (4 * d + 4 + 4 * (d + 1))    # points in, ids out, the stored record
        by += b * 4 + b * 4                    # ids to erase, their marks
    if case["kind"] == "build":
        by += n * (4 * d + 4 + 4 * (d + 1))
    return {"bytes": float(by), "flops": float(fl)}


def tolerance(case):
    return "exact"


def _brute(points, ids, queries, k):
    """The k nearest of `points` (ids ascending) per query by (d2, id), padded as kNN is."""
    m, dim, piece = queries.shape[0], queries.shape[1], 1 << 16
    oi = torch.full((m, k), -1, dtype=torch.int32, device="cuda")
    od = torch.full((m, k), torch.iinfo(torch.int64).max, dtype=torch.int64, device="cuda")
    for a in range(0, m, 2048):
        q = queries[a:a + 2048].to(torch.int64)
        bd, bi = od[a:a + 2048], oi[a:a + 2048]
        for p in range(0, points.shape[0], piece):
            pts = points[p:p + piece].to(torch.int64)
            # d2 < 16 * 2^40 and the place in the piece < 2^16: one word orders both
            key = torch.zeros(q.shape[0], pts.shape[0], dtype=torch.int64, device="cuda")
            for c in range(dim):
                g = q[:, c:c + 1] - pts[:, c]
                key.addcmul_(g, g)
            key = key.mul_(1 << 16).add_(torch.arange(pts.shape[0], device="cuda"))
            key = key.topk(min(k, pts.shape[0]), largest=False, sorted=True).values
            # earlier pieces hold smaller ids, so a stable sort by d2 keeps ties by id
            d = torch.cat([bd, key >> 16], 1)
            i = torch.cat([bi, ids[p + (key & 0xFFFF)]], 1)
            d, o = d.sort(dim=1, stable=True)
            bd, bi = d[:, :k], i.gather(1, o)[:, :k]
        od[a:a + 2048], oi[a:a + 2048] = bd, bi
    return oi, od


def exact(case, seed):
    kind, k = case["kind"], case["k"]
    if kind == "forests":
        n, b, m = _forest_sizes(case)
        if sum(x * y for x, y in zip(n, m)) > EXACT_PAIRS or len(n) > 64:
            return None
        w = _Many(case, seed)
        pts, gone = _fresh(w.batches[0], 0).split(w.b), w.out[0].split(w.b)
        new, oi, od, first = [], [], [], 0
        for j in range(len(n)):
            keep = torch.ones(n[j] + b[j], dtype=torch.bool, device="cuda")
            keep[gone[j] - first] = False
            first += n[j]
            ids = torch.nonzero(keep).flatten().to(torch.int32)
            x, y = _brute(torch.cat([w.points[j], pts[j]])[keep], ids, w.queries[j], k)
            new.append(torch.arange(n[j], n[j] + b[j], dtype=torch.int32, device="cuda"))
            oi.append(x)
            od.append(y)
        return {"new": torch.cat(new), "erased": torch.tensor(b), "ids": torch.cat(oi), "d2": torch.cat(od)}
    if float(case["n"]) * case["queries"] > EXACT_PAIRS:
        return None
    w = _World(case, seed)
    every, total = [w.points], case["n"]
    live = torch.arange(total, dtype=torch.int32, device="cuda")
    updates = list(w.churn)
    if kind == "step":
        updates.append((_fresh(w.batches[0], 0), w.out[0]))
    new = live.clone()
    for pts, gone in updates:
        new = torch.arange(total, total + pts.shape[0], dtype=torch.int32, device="cuda")
        total += pts.shape[0]
        every.append(pts)
        live[gone] = new
    ids = live.sort().values
    oi, od = _brute(torch.cat(every)[ids.long()], ids, w.queries, k)
    got = {"ids": oi, "d2": od}
    if kind in ("step", "build"):
        got["new"] = new
    if kind == "step":
        got["erased"] = case["batch"]
    return got
