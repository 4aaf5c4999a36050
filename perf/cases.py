"""Performance cases: what users of the library have it do, through its public Python entry points.

A case is one call a program makes: a batch of range-filtered k-NN queries (`Index.search` on device tensors,
`Index.search_host` on host arrays), the exact filtered scan (`Index.exact_search`, used for ground truth and for
pre-filtering), or a (re)build of an index followed by opening it and answering the first batch.  Data are
seeded low-rank mixtures like those of the repository's workloads: byte-valued descriptors ("bytes"),
unit-length embeddings ("unit"), unit-length embeddings whose attribute is an insertion time correlated with the
cluster ("timeline") and anisotropic text-like vectors ("text").  Range widths are log-uniform between
2^-min_log2 and 1 of the objects, the mixed selectivity of the repository's benchmark.
"""
import os
import tempfile

import numpy as np
import torch

import paper_2608_16491_b200 as frog

DEFAULT_BUDGET = 16          # expansion budget of a call without parameters


def _case(name, op, data, n, d, nq, k, beam=0, budget=0, storage="f32", min_log2=10):
    return dict(name=name, op=op, data=data, n=n, d=d, nq=nq, k=k, beam=beam, budget=budget, storage=storage,
                min_log2=min_log2)


def listed():
    return [
        # One interactive query against a resident index: the latency a single user sees.
        _case("one-query", "search", "bytes", 100_000, 128, 1, 10, beam=64, budget=64, min_log2=3),
        # A handful of requests collected by a server, NumPy arrays in and pinned arrays out, default parameters.
        _case("few-hosted", "host", "unit", 100_000, 96, 16, 10, beam=64),
        # A micro-batch of an online service: fewer queries than the GPU has warps.
        _case("micro-batch", "search", "unit", 200_000, 96, 250, 10, beam=32, budget=64),
        # The throughput batch of the repository's benchmark (10,000 queries, recall-tuned beam and budget).
        _case("batch-bytes", "search", "bytes", 400_000, 128, 10_000, 10, beam=44, budget=64),
        # Candidate generation: long result lists (k = 100) for a large batch.
        _case("batch-top100", "search", "unit", 400_000, 96, 10_000, 100, beam=112, budget=64),
        # Recent-items queries: attribute correlated with content, needs wide beams and large budgets.
        _case("batch-timeline", "search", "timeline", 100_000, 96, 3_000, 10, beam=160, budget=128, min_log2=7),
        # Long text embeddings, 3 KB a row.
        _case("batch-text", "search", "text", 20_000, 768, 2_000, 10, beam=192, budget=128, min_log2=7),
        # A row length that is neither short nor a power of two, and a caller that keeps the default budget.
        _case("ragged-rows", "search", "unit", 100_000, 100, 1_001, 10, beam=128, min_log2=9),
        # Half-precision rows.
        _case("half-rows", "search", "bytes", 100_000, 128, 5_000, 10, beam=64, budget=64, storage="f16"),
        # Exact answers for a few queries over all ranges (a pre-filtering fall-back while serving).
        _case("exact-few", "exact", "unit", 400_000, 96, 6, 10, min_log2=8),
        # Ground truth for a validation set.
        _case("exact-truth", "exact", "bytes", 100_000, 128, 2_000, 100),
        # Rebuilding a shard, opening it and answering its first batch.
        _case("rebuild", "build", "unit", 100_000, 96, 200, 10, beam=32, budget=64, min_log2=8),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(2 ** rng.uniform(np.log2(lo), np.log2(hi))))

    op = rng.choice(["search"] * 6 + ["host", "exact", "exact", "build"])
    data = rng.choice(["bytes", "unit", "unit", "timeline", "text"])
    d = {"bytes": 128, "text": rng.choice([384, 768])}.get(data) or rng.choice([96, 96, 32, 50, 64, 100, 128, 200])
    n = log(5_000, 20_000 if data == "text" else 100_000)
    k = rng.choice([1, 10, 10, 10, 50, 100])
    if op == "exact":
        nq = log(1, 2_000)
        return _case(None, op, data, n, d, nq, k, min_log2=rng.choice([4, 7, 10]))
    nq = log(1, {"search": 10_000, "host": 2_000, "build": 500}[op])
    if data == "text":
        nq = max(1, nq // 5)
    if op == "build":
        n = min(n, 5_000 if data == "text" else 80_000)
    beam = max(k, log(16, 192))
    budget = rng.choice([0, 16, 32, 64, 64, 96, 128])
    storage = rng.choice(["f32", "f32", "f32", "f16"]) if op == "search" else "f32"
    return _case(None, op, data, n, d, nq, k, beam=beam, budget=budget, storage=storage, min_log2=rng.choice([7, 10]))


# ---- inputs ----------------------------------------------------------------------------------------------
def _mixture(g, labels, centers, loads, noise):
    """x_i = center + z_i loading + e_i for cluster labels[i] (on the GPU)."""
    n, d, r = labels.shape[0], centers.shape[1], loads.shape[1]
    x = torch.randn(n, d, generator=g, device="cuda") * noise
    z = torch.randn(n, r, generator=g, device="cuda")
    order = torch.argsort(labels, stable=True)
    bounds = torch.searchsorted(labels[order], torch.arange(centers.shape[0] + 1, device="cuda")).tolist()
    for c in range(centers.shape[0]):
        rows = order[bounds[c]:bounds[c + 1]]
        x[rows] += centers[c] + z[rows] @ loads[c]
    return x


def _vectors(case, g):
    """(base vectors, attributes, queries) on the GPU."""
    n, d, nq, data = case["n"], case["d"], case["nq"], case["data"]

    def rand(size, high):
        return torch.randint(0, high, (size,), generator=g, device="cuda")

    if data == "text":
        sd = torch.arange(1, d + 1, device="cuda", dtype=torch.float64).pow(-0.4).float()
        base, queries = (torch.randn(c, d, generator=g, device="cuda") * sd for c in (n, nq))
    else:
        clusters, s_c, s_l, s_e = (64, 20.0, 34.4, 4.0) if data == "bytes" else (128, 0.5, 1.0, 0.12)
        centers = torch.randn(clusters, d, generator=g, device="cuda") * s_c
        loads = torch.randn(clusters, 12, d, generator=g, device="cuda") * (s_l / 12 ** 0.5)
        labels = rand(n, clusters)
        if data == "timeline":          # clusters arrive in contiguous blocks of the timeline
            blocks = rand(1024, clusters)
            labels = blocks[torch.arange(n, device="cuda") * 1024 // n]
        base = _mixture(g, labels, centers, loads, s_e)
        queries = _mixture(g, rand(nq, clusters), centers, loads, s_e)
    if data == "bytes":
        base, queries = base.abs().round().clamp(0, 255), queries.abs().round().clamp(0, 255)
    else:
        base, queries = (x / x.norm(dim=1, keepdim=True) for x in (base, queries))
    attrs = torch.arange(n, device="cuda") if data == "timeline" else rand(n, 1_000_000 if data == "bytes" else 2**31 - 1)
    return base.contiguous(), attrs.to(torch.int32), queries.contiguous()


def _ranges(case, g, attrs):
    """[lo, hi] of each query: w consecutive objects in attribute order at a uniform place."""
    n, nq = case["n"], case["nq"]
    u = torch.rand(2, nq, generator=g, device="cuda", dtype=torch.float64)
    w = (n * torch.exp2(-case["min_log2"] * u[0])).round().long().clamp(1, n)
    start = torch.minimum((u[1] * (n - w + 1)).long(), n - w)
    ordered = attrs.sort().values
    return ordered[start].contiguous(), ordered[start + w - 1].contiguous()


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    base, attrs, queries = _vectors(case, g)
    lo, hi = _ranges(case, g, attrs)
    base, attrs = base.cpu().numpy(), attrs.cpu().numpy()
    params = frog.Params(budget=case["budget"], storage=frog.STORAGE_F16 if case["storage"] == "f16" else frog.STORAGE_F32)
    state = dict(case=case, params=params if case["budget"] or case["storage"] == "f16" else None)
    folder = tempfile.TemporaryDirectory()
    path = os.path.join(folder.name, "index")
    if case["op"] == "build":
        return dict(state, folder=folder, path=path, base=base, attrs=attrs, queries=queries, lo=lo, hi=hi)
    # the exact scan reads no graph: a minimal one is made quickly
    quick = dict(m=4, ef_c=4, patience=1, n_inv=8) if case["op"] == "exact" else {}
    frog.build_index_gpu(base, attrs, path, **quick)
    index = frog.Index.load(path)
    folder.cleanup()
    if case["storage"] == "f16":
        index.enable_f16()
    if case["op"] == "host":
        queries, lo, hi = (x.cpu().numpy() for x in (queries, lo, hi))
    return dict(state, index=index, queries=queries, lo=lo, hi=hi)


def run(state):
    case = state["case"]
    k, beam = case["k"], case["beam"]
    if case["op"] == "build":
        frog.build_index_gpu(state["base"], state["attrs"], state["path"])
        index = frog.Index.load(state["path"])
        ids, dists = index.search(state["queries"], state["lo"], state["hi"], k, beam, params=state["params"])
        index.close()
        return ids, dists, np.fromfile(state["path"], dtype=np.uint8)
    index, args = state["index"], (state["queries"], state["lo"], state["hi"], k)
    if case["op"] == "exact":
        return index.exact_search(*args)
    if case["op"] == "host":
        return index.search_host(*args, beam, params=state["params"])
    return index.search(*args, beam, params=state["params"])


# ---- what a pass cannot do without -----------------------------------------------------------------------
def _mean_width(case):
    """Mean number of objects in a range (log-uniform fractions)."""
    a = case["min_log2"] * np.log(2.0)
    return case["n"] * (1 - np.exp(-a)) / a


def work(case):
    n, d, nq, k, beam = case["n"], case["d"], case["nq"], case["k"], case["beam"]
    row = (2 if case["storage"] == "f16" else 4) * d
    m = 16 if d <= 300 else 32
    layers = max(1, int(np.ceil(np.log2(n))) + 1 - (7 if d <= 300 else 6))
    io = nq * (4 * d + 8 + 8 * k)
    width = _mean_width(case)
    if case["op"] == "exact":
        # every object of a range is compared; a row that several ranges share is read once
        return {"bytes": int(io + min(nq * width, n) * (row + 8)), "flops": int(nq * width * 3 * d)}
    # a beam search expands at least its beam; an expansion reads about three rows of m candidates and
    # evaluates a fifth to a third of those the budget admits (measured: the rest have been seen)
    expansions = min(beam, width)
    evaluated = min(expansions * max(4, min(case["budget"] or DEFAULT_BUDGET, 3 * m) / 4), width)
    graph = nq * expansions * 3 * m * 4
    rows = nq * evaluated
    search = {"bytes": int(io + min(graph, n * layers * m * 4) + min(rows, n) * row), "flops": int(rows * 3 * d)}
    if case["op"] != "build":
        return search
    # per object and layer: about ef_c candidates reached on the sibling side, 64 pairs of the candidates kept;
    # vectors in, vectors and graph out
    ef_c = 128 if d <= 300 else 256
    return {"bytes": int(search["bytes"] + n * (3 * 4 * d + 2 * layers * m * 4)),
            "flops": int(search["flops"] + n * layers * (ef_c * 4 + 64 * m) * 3 * d)}


def tolerance(case):
    """The order of every sum and every tie rule is part of the interface (ids, distance bits and index files are
    pinned against an independent implementation), so results are equal bit for bit."""
    return "exact"
