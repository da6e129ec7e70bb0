"""What this repository's speed is measured on: index builds, insertions,
batched searches and exact k-NN, each through the package's public entry
points, over the sizes that its workloads, tests and benchmark use.

A case is a dict of plain values with a "kind":
  search  one call of Index.search on an index built beforehand
  build   Index(...) and the graphs it made, read back layer by layer
  insert  an index built on the first points, the others appended in batches
  knn     one call of exact_knn
"""
import math

import torch

import paper_2505_17368_gb300 as henn

METRIC = {"l2": henn.L2, "angular": henn.ANGULAR}
STORAGE = {"f32": henn.F32, "bf16": henn.BF16, "fp8": henn.FP8E4M3}
GRAPH = {"nsw": henn.GRAPH_NSW, "knn": henn.GRAPH_KNN}

# How a search goes through the upper layers.  greedy: Alg. 4.  walk: a beam
# on every layer.  tiles / sort: the lowest layer of at most so many points
# gives its exact candidates, which seed narrow beams below it.
UPPER = {
    "greedy": dict(ef_upper=1),
    "walk": dict(ef_upper=32),
    "tiles": dict(ef_upper=16, descend_all=1, ef_l1=8, exact_upper=8192, exact_method=henn.EXACT_TILES),
    "sort": dict(ef_upper=16, descend_all=1, exact_upper=512, exact_method=henn.EXACT_SORT),
}


def _search(name, data, n, d, nq, k, ef, storage, metric="l2", upper="greedy", mixed=False, host=False):
    c = dict(kind="search", data=data, n=n, d=d, nq=nq, k=k, ef=ef, storage=storage, metric=metric, upper=upper,
             mixed=mixed, host=host)
    return dict(c, name=name) if name else c


def _build(name, data, n, d, storage, metric="l2", graph="nsw"):
    c = dict(kind="build", data=data, n=n, d=d, storage=storage, metric=metric, graph=graph)
    return dict(c, name=name) if name else c


def _insert(name, data, n, d, add, batch, storage, metric="l2"):
    c = dict(kind="insert", data=data, n=n, d=d, add=add, batch=batch, storage=storage, metric=metric)
    return dict(c, name=name) if name else c


def _knn(name, data, n, d, nq, k, metric="l2"):
    c = dict(kind="knn", data=data, n=n, d=d, nq=nq, k=k, metric=metric)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one query per call, as a program does that answers a user's request
        # at once (and as the paper times its queries): latency
        _search("search-one", "exponential", 50_000, 32, 1, 10, 64, "f32"),
        # a small batch against the benchmark's index: a service that
        # collects requests for a moment
        _search("search-64", "mixture", 1_000_000, 128, 64, 10, 64, "bf16", upper="walk"),
        # the benchmark's batch: SIFT-sized vectors in BF16, 10,000 queries,
        # the exact layer from distance tiles
        _search("search-10k", "mixture", 1_000_000, 128, 10_000, 10, 50, "bf16", upper="tiles"),
        # word vectors with cosine distance, rows that are no multiple of a
        # line, FP8 rows, and 100 results a query: candidates for a re-ranker
        _search("search-angular-k100", "mixture", 50_000, 100, 1_000, 100, 200, "fp8", "angular", "walk"),
        # wide vectors (images, text embeddings) in BF16
        _search("search-wide", "mixture", 100_000, 960, 2_000, 10, 128, "bf16", upper="tiles"),
        # requests of several users in one call, each with its own number of
        # results and beam width, in ordinary host arrays
        _search("search-mixed-host", "shells", 200_000, 64, 5_000, 100, 512, "f32", mixed=True, host=True),
        # an index made on the fly for a small set
        _build("build-10k", "uniform", 10_000, 32, "f32"),
        # the benchmark's index
        _build("build-1m", "mixture", 1_000_000, 128, "bf16"),
        # an index of wide vectors
        _build("build-wide", "mixture", 100_000, 960, "bf16"),
        # an index that grows: two batches of new points
        _insert("insert-20k", "mixture", 100_000, 128, 20_000, 10_000, "bf16"),
        # exact neighbours of the benchmark's queries: the ground truth that
        # recall is scored against
        _knn("knn-10k", "mixture", 1_000_000, 128, 10_000, 10),
        # exact neighbours by cosine distance, 100 of them, of a small batch
        _knn("knn-k100", "mixture", 50_000, 100, 1_000, 100, "angular"),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["search", "search", "search", "build", "build", "insert", "knn", "knn"])
    metric = rng.choice(["l2", "l2", "angular"])
    storage = rng.choice(["f32", "bf16", "bf16", "fp8"])
    if metric == "angular":
        data = "mixture"
    else:
        data = rng.choice(["mixture", "mixture", "exponential", "uniform", "shells"])
    if kind == "search":
        d = log(16, 960)
        n = min(log(2_000, 1_000_000), int(128e6 / d))
        mixed = rng.random() < 0.25
        k = 100 if mixed else rng.choice([1, 10, 10, log(2, 100)])
        ef = 512 if mixed else max(k, log(16, 256))
        nq = log(1, 10_000)
        upper = rng.choice(["greedy", "walk", "tiles"] + (["sort"] if n >= 10_000 else []))
        return _search(None, data, n, d, nq, k, ef, storage, metric, upper, mixed, rng.random() < 0.25)
    if kind == "build":
        d = log(16, 960)
        n = min(log(2_000, 500_000), int(32e6 / d))
        return _build(None, data, n, d, storage, metric, rng.choice(["nsw", "nsw", "knn"]))
    if kind == "insert":
        d = log(16, 512)
        n = min(log(5_000, 200_000), int(16e6 / d))
        add = log(1, max(2, n // 5))
        return _insert(None, data, n, d, add, max(1, add // rng.choice([1, 2, 3])), storage, metric)
    d = log(16, 960)
    n = min(log(2_000, 1_000_000), int(128e6 / d))
    return _knn(None, data, n, d, log(1, 10_000), rng.choice([1, 10, 10, log(2, 112)]), metric)


# ------------------------------------------------------------------ inputs


def _points(data, n, d, g, base):
    """n rows of FP32 on the GPU; base: the index's points, else queries of the same distribution."""
    dev = g.device
    if data == "uniform":
        return torch.rand(n, d, generator=g, device=dev)
    if data == "exponential":
        return torch.empty(n, d, device=dev).exponential_(4.0, generator=g)
    if data == "shells":  # points on spheres of radius 2^-i, shell after shell; queries near the innermost
        x = torch.randn(n, d, generator=g, device=dev)
        x /= x.norm(dim=1, keepdim=True)
        if base:
            return x * torch.exp2(-torch.div(torch.arange(n, device=dev) * 20, n, rounding_mode="floor"))[:, None]
        return x * torch.exp2(-20.0 + 2.0 * torch.rand(n, 1, generator=g, device=dev))
    raise ValueError(data)


def _inputs(case, seed, nq):
    """The index's points and the queries (mixture: clusters of one seed, values about 0 .. 255 as SIFT's are)."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    n, d, data = case["n"] + case.get("add", 0), case["d"], case["data"]
    if data != "mixture":
        return _points(data, n, d, g, True), _points(data, nq, d, g, False)
    clusters = max(8, n // 1000)
    centre = torch.randn(clusters, d, generator=g, device=dev)
    sigma = 0.1 + 0.4 * torch.rand(clusters, generator=g, device=dev)
    out = []
    for m in (n, nq):
        c = torch.randint(clusters, (m,), generator=g, device=dev)
        x = torch.randn(m, d, generator=g, device=dev)
        x.mul_(sigma[c, None]).add_(centre[c]).mul_(23.0).add_(127.5)
        out.append(x if case["metric"] == "l2" else (x - 127.5) / 23.0)
    return out


def _index(case, X):
    return henn.Index(X, metric=METRIC[case["metric"]], storage=STORAGE[case["storage"]],
                      graph=GRAPH[case.get("graph", "nsw")], seed=1)


def prepare(case, seed):
    X, Q = _inputs(case, seed, case.get("nq", 1))
    if case["kind"] != "search":
        return dict(case=case, X=X, Q=Q)
    k, ef = case["k"], case["ef"]
    if case["mixed"]:
        g = torch.Generator(device=X.device)
        g.manual_seed(seed + 1)
        u = torch.rand(case["nq"], generator=g, device=X.device)
        ef = torch.exp(math.log(32) + (math.log(512) - math.log(32)) * u).round().to(torch.int32)
        k = torch.where(torch.rand(case["nq"], generator=g, device=X.device) < 0.5, 10, 100).to(torch.int32)
    if case["host"]:
        Q = Q.cpu().numpy()
        if case["mixed"]:
            k, ef = k.cpu().numpy(), ef.cpu().numpy()
    return dict(case=case, index=_index(case, X), Q=Q, k=k, ef=ef)


# -------------------------------------------------------------------- runs


def _layers(index):
    return [index.layer(i) for i in range(len(index.info()["sizes"]))]


def run(state):
    case = state["case"]
    if case["kind"] == "search":
        ids, dists, _ = state["index"].search(state["Q"], k=state["k"], ef=state["ef"],
                                              out_stride=case["k"], **UPPER[case["upper"]])
        return {"ids": ids, "dists": dists}
    if case["kind"] == "knn":
        ids, dists = henn.exact_knn(state["X"], state["Q"], case["k"], metric=METRIC[case["metric"]])
        return {"ids": ids, "dists": dists}
    X, n = state["X"], case["n"]
    index = _index(case, X[:n])
    for r in range(n, n + case.get("add", 0), case.get("batch", 1)):
        index.insert(X[r:min(r + case["batch"], X.shape[0])])
    out = _layers(index)
    index.close()
    return out


# -------------------------------------------------------------------- work


def work(case):
    """Each input read once and each output written once.  A search reads, of the index, at least the rows and the
    links of the points that its beam ends with, and never more than the whole index; a build and an insertion
    compare each point with those before it (kNN graph: with all others)."""
    n, d = case["n"], case["d"]
    if case["kind"] == "search":
        nq = case["nq"]
        k, ef = (55, 173) if case["mixed"] else (case["k"], max(case["k"], case["ef"]))  # the means where mixed
        row = d * {"f32": 4, "bf16": 2, "fp8": 1}[case["storage"]] + 32 * 4
        return {"bytes": nq * (4 * d + 12 * case["k"]) + min(nq * ef, n) * row, "flops": 3.0 * d * nq * max(k, ef)}
    if case["kind"] == "knn":
        nq = case["nq"]
        return {"bytes": 4 * d * (n + nq) + 12 * nq * case["k"], "flops": 2.0 * d * n * nq}
    m = n + case.get("add", 0)
    pairs = m * (m - 1) / (1 if case.get("graph") == "knn" else 2)
    # links in (16 int32 and 16 float32) and 32 int32 out a point, the upper layers a fifteenth more
    return {"bytes": 4 * d * m + m * 64 * 4 * 16 / 15, "flops": 2.0 * d * pairs}


def exact(case, seed):
    """Exact neighbours' distances in 64 bits (ids are left out: two distances may tie in 32 bits).  A walk's answer
    and a graph's links have no such value: which points they hold follows from comparisons made in 32 bits."""
    if case["kind"] != "knn":
        return None
    X, Q = _inputs(case, seed, case["nq"])
    X, Q = X.double(), Q.double()
    if case["metric"] == "angular":
        X /= X.norm(dim=1, keepdim=True)
        Q /= Q.norm(dim=1, keepdim=True)
    k, n = case["k"], case["n"]
    kk = min(k, n)
    xx = (X * X).sum(1)
    found = []
    rows = max(1, min(512, int(1e9 / n)))
    for r in range(0, Q.shape[0], rows):
        q = Q[r:r + rows]
        near = torch.topk((q * q).sum(1)[:, None] + xx - 2.0 * (q @ X.T), min(n, kk + 8), largest=False).indices
        dd = ((X[near] - q[:, None, :]) ** 2).sum(2).sort(dim=1).values[:, :kk]
        found.append(0.5 * dd if case["metric"] == "angular" else dd.sqrt())
    dists = torch.cat(found)
    if kk < k:
        dists = torch.cat([dists, torch.full((dists.shape[0], k - kk), math.inf, dtype=dists.dtype, device=dists.device)], 1)
    return {"ids": None, "dists": dists}
