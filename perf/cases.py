"""The work that programs built on this library have it do, as cases to time.

Every case is one call chain through the public entry points (the binding of
include/simjoin.h), from points on the GPU to results on the GPU:

* ``pairs``   sj_build_index, sj_self_join, sj_result_copy: the similarity
              self-join itself.  The pair list comes back as a set in no
              particular order; the program makes of it what a graph is kept
              as: an adjacency matrix for a small set of points, else the
              ordered pair list, in a buffer of fixed capacity.
* ``dbscan``  the join, then sj_dbscan on its result: the labels of all points.
* ``knn``     the join with distances, then sj_knn_from_join: neighbour
              indices and distances of all points.
* ``batch``   sj_join_batch: many small independent joins in one call, the
              ordered pairs of all of them.

A case gives the sizes; the points are drawn from the seed (the distributions
of workloads.py, and Gaussian clusters over uniform noise in low dimension,
the usual shape of data that is clustered by density).
"""
import ctypes
import json
import math

import torch

from paper_2209_11287_gb300 import binding, workloads

DEV = "cuda"


def listed():
    return [
        # a few hundred to a few thousand points, joined on demand (a small
        # table, one frame of detections): all latency and launches
        {"name": "pairs_2d_1500", "kind": "pairs", "data": "uniform", "n": 1500, "d": 2, "neighbours": 32},
        # the small planar workload of the benchmark
        {"name": "pairs_2d_16384", "kind": "pairs", "data": "uniform", "n": 16384, "d": 2, "neighbours": 32},
        # near-duplicates of a large 4-D catalogue: few neighbours, a key space
        # too large for the counting sort
        {"name": "pairs_4d_1m", "kind": "pairs", "data": "uniform", "n": 1_000_001, "d": 4, "neighbours": 4},
        # the plain FP64 tile that the paper is about, with the distances
        {"name": "knn_4d_fp64", "kind": "knn", "data": "uniform", "n": 200_000, "d": 4, "neighbours": 64, "k": 8,
         "kernel": "fp64_fma"},
        # the 2M x 4-D headline workload, its neighbourhoods used for density
        # clustering
        {"name": "dbscan_4d_2m", "kind": "dbscan", "data": "uniform", "n": 2_000_000, "d": 4, "neighbours": 64,
         "min_pts": 64},
        # density clustering of a 3-D point set (odd dimension, ragged size)
        {"name": "dbscan_3d_clusters", "kind": "dbscan", "data": "clusters", "n": 700_003, "d": 3, "neighbours": 24,
         "min_pts": 10},
        # neighbours of a 3-D point cloud (normals, features)
        {"name": "knn_3d", "kind": "knn", "data": "uniform", "n": 200_003, "d": 3, "neighbours": 48, "k": 16},
        # neighbours of 16-D descriptors
        {"name": "knn_16d", "kind": "knn", "data": "mixture16d", "n": 100_000, "d": 16, "k": 32},
        # the larger workloads of the benchmark: 16-D Gaussian mixture
        # (clustered), 64-D clipped exponential (nearly all pairs are
        # candidates), and 16-D without an index (the paper's brute-force
        # comparison)
        {"name": "dbscan_mixture16d", "kind": "dbscan", "data": "mixture16d", "n": 500_000, "d": 16, "min_pts": 32},
        {"name": "pairs_expo64d", "kind": "pairs", "data": "expo64d", "n": 200_000, "d": 64},
        {"name": "brute_16d", "kind": "pairs", "data": "brute16d", "n": 1 << 17, "d": 16, "index": False},
        # a request's worth of independent joins of mixed size and dimension
        {"name": "batch_96", "kind": "batch", "first": 0, "count": 96},
    ]


def _log_size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pairs", "pairs", "low", "low", "fp64", "dbscan", "dbscan", "dbscan16", "knn", "knn16", "expo",
                       "brute", "batch"])
    if kind == "pairs":  # planar and small
        return {"kind": "pairs", "data": "uniform", "n": _log_size(rng, 300, ADJACENCY), "d": rng.choice([2, 2, 3]),
                "neighbours": rng.randint(8, 64)}
    if kind == "low":
        return {"kind": "pairs", "data": "uniform", "n": _log_size(rng, 20_000, 1_000_000),
                "d": rng.choice([2, 3, 4, 5]), "neighbours": rng.randint(2, 8)}
    if kind == "fp64":
        return {"kind": "knn", "data": "uniform", "n": _log_size(rng, 5_000, 200_000), "d": rng.choice([2, 3, 4]),
                "neighbours": rng.randint(16, 64), "k": rng.randint(4, 16), "kernel": "fp64_fma"}
    if kind == "dbscan":
        n = _log_size(rng, 50_000, 1_500_000)
        if rng.random() < 0.33:
            neighbours = rng.randint(12, 64)
            return {"kind": "dbscan", "data": "uniform", "n": n, "d": rng.choice([2, 3, 4]), "neighbours": neighbours,
                    "min_pts": neighbours}
        return {"kind": "dbscan", "data": "clusters", "n": n, "d": rng.choice([2, 3, 4]),
                "neighbours": rng.randint(12, 40), "min_pts": rng.randint(4, 12)}
    if kind == "dbscan16":
        return {"kind": "dbscan", "data": "mixture16d", "n": _log_size(rng, 30_000, 500_000), "d": 16,
                "min_pts": rng.randint(16, 48)}
    if kind == "knn":
        return {"kind": "knn", "data": rng.choice(["uniform", "clusters"]), "n": _log_size(rng, 10_000, 250_000),
                "d": rng.choice([2, 3, 4]), "neighbours": rng.randint(24, 64), "k": rng.randint(4, 24)}
    if kind == "knn16":
        return {"kind": "knn", "data": "mixture16d", "n": _log_size(rng, 20_000, 120_000), "d": 16,
                "k": rng.randint(8, 40)}
    if kind == "expo":
        return {"kind": "pairs", "data": "expo64d", "n": _log_size(rng, 25_000, 200_000), "d": 64}
    if kind == "brute":
        return {"kind": "pairs", "data": "brute16d", "n": _log_size(rng, 25_000, 1 << 17), "d": 16, "index": False}
    return {"kind": "batch", "first": rng.randint(0, 3900), "count": _log_size(rng, 24, 96)}


# up to this many points the graph is kept as an adjacency matrix
ADJACENCY = 20_000
CLUSTERS, SIGMA, NOISE = 64, 0.02, 0.1


def _neighbours(case):
    """Mean neighbours (the point itself left out) that the case's eps is set for."""
    return {"mixture16d": 100.0, "expo64d": 50.0, "brute16d": 50.0}.get(case.get("data"), case.get("neighbours", 32))


def _points(case, seed):
    """(points on the GPU, eps)."""
    n, d, data = case["n"], case["d"], case["data"]
    if data in workloads.CONFIGS:
        w = workloads.CONFIGS[data](n=n, seed=seed)
        return torch.from_numpy(w.points).to(DEV), w.eps
    g = torch.Generator(device=DEV).manual_seed(seed)
    if data == "uniform":
        return torch.rand((n, d), dtype=torch.float64, device=DEV, generator=g), workloads.ball_eps(n, d, case["neighbours"])
    # Gaussian clusters over uniform noise; eps for the mean over the clusters'
    # points of the neighbours in their own cluster: two points of a cluster
    # differ by N(0, 2 sigma^2), of density (4 pi sigma^2)^(-d/2) near 0
    centres = torch.rand((CLUSTERS, d), dtype=torch.float64, device=DEV, generator=g)
    label = torch.randint(0, CLUSTERS, (n,), device=DEV, generator=g)
    x = centres[label] + SIGMA * torch.randn((n, d), dtype=torch.float64, device=DEV, generator=g)
    noise = torch.rand((n,), dtype=torch.float64, device=DEV, generator=g) < NOISE
    x = torch.where(noise[:, None], torch.rand((n, d), dtype=torch.float64, device=DEV, generator=g), x).contiguous()
    per = (1.0 - NOISE) * n / CLUSTERS
    ball = math.pi ** (d / 2) / math.gamma(d / 2 + 1)
    return x, (case["neighbours"] * (4 * math.pi * SIGMA ** 2) ** (d / 2) / (per * ball)) ** (1.0 / d)


def _batch_sizes(case):
    return [(i,) + workloads.batch_instance_params(i)[:2] for i in range(case["first"], case["first"] + case["count"])]


def _batch_eps(sizes):
    with open(workloads.EPS_TABLE) as f:
        stored = json.load(f).get("batched", {})
    return [float(stored.get(str(i), workloads.ball_eps(n, d, 32.0))) for i, n, d in sizes]


def _capacity(case):
    """Pairs that the program's buffer holds: the mean its eps is set for, the
    points themselves, and room for what differs from one set to the next."""
    if case["kind"] == "batch":
        return sum(int(45 * n) + 4096 for _, n, _ in _batch_sizes(case))
    return int(1.25 * case["n"] * (_neighbours(case) + 1)) + 4096


def prepare(case, seed):
    if case["kind"] == "batch":
        g = torch.Generator(device=DEV).manual_seed(seed)
        sizes = _batch_sizes(case)
        pts = [torch.rand((n, d), dtype=torch.float64, device=DEV, generator=g) for _, n, d in sizes]
        return {"case": case, "points": pts, "inputs": binding.BatchInputs(pts, _batch_eps(sizes)),
                "options": binding.sj_default_options(), "capacity": _capacity(case)}
    x, eps = _points(case, seed)
    opt = binding.sj_default_options(
        kernel=case.get("kernel", "auto"), emit_distances=int(case["kind"] == "knn"),
        indexed_dims=0 if case.get("index", True) else binding.SJ_NO_INDEX)
    return {"case": case, "points": x, "eps": eps, "options": opt, "capacity": _capacity(case)}


def _ordered(keys, capacity):
    """The 64-bit pairs as a list of fixed capacity: ordered, -1 past the last."""
    if keys.numel() > capacity:
        raise RuntimeError(f"{keys.numel()} pairs, room for {capacity}")
    out = torch.empty(capacity, dtype=torch.int64, device=DEV)
    out[:keys.numel()] = torch.unique(keys)
    out[keys.numel():] = -1
    return out.view(torch.int32).view(-1, 2)


def _run_pairs(result, n, capacity):
    pairs = torch.empty((result.count, 2), dtype=torch.int32, device=DEV)
    binding.sj_result_copy(result, pairs)
    if n <= ADJACENCY:
        at = pairs[:, 0].long() * n + pairs[:, 1]
        return {"adjacency": torch.zeros(n * n, dtype=torch.uint8, device=DEV).index_fill_(0, at, 1).view(n, n)}
    # one 64-bit key a pair, (j, i): the pairs ordered by j, then i
    return {"pairs": _ordered(pairs.view(torch.int64).view(-1), capacity), "count": result.count}


def _run_dbscan(result, n, min_pts):
    labels = torch.empty(n, dtype=torch.int32, device=DEV)
    clusters = ctypes.c_int64(0)
    # the C entry point itself: its outputs may stay on the GPU
    if binding.load().sj_dbscan(ctypes.byref(result), n, min_pts, labels.data_ptr(), ctypes.byref(clusters)):
        raise RuntimeError(binding.sj_last_error_message())
    return {"labels": labels, "clusters": clusters.value}


def _run_knn(result, n, k):
    idx = torch.empty((n, k), dtype=torch.int32, device=DEV)
    dist = torch.empty((n, k), dtype=torch.float64, device=DEV)
    found = torch.empty(n, dtype=torch.int32, device=DEV)
    if binding.load().sj_knn_from_join(ctypes.byref(result), n, k, idx.data_ptr(), dist.data_ptr(), found.data_ptr()):
        raise RuntimeError(binding.sj_last_error_message())
    return {"idx": idx, "dist": dist, "found": found}


def _run_batch(state):
    res = binding.sj_join_batch_raw(state["inputs"], state["options"])
    try:
        counts = [int(r.count) for r in res]
        pairs = torch.empty((sum(counts), 2), dtype=torch.int32, device=DEV)
        at = 0
        for r, c in zip(res, counts):
            binding.sj_result_copy(r, pairs[at:at + c])
            at += c
    finally:
        binding.sj_results_free(res)
    counts = torch.tensor(counts, dtype=torch.int64).to(DEV)
    # the instances have at most 65536 points, so bits 16 .. of a pair's first
    # index take the instance's number: pairs ordered by j, instance, i
    inst = torch.arange(counts.numel(), device=DEV).repeat_interleave(counts, output_size=pairs.shape[0])
    return {"pairs": _ordered(pairs.view(torch.int64).view(-1) + (inst << 16), state["capacity"]), "counts": counts}


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        return _run_batch(state)
    h = binding.sj_build_index(state["points"], state["eps"], state["options"])
    try:
        r = binding.sj_self_join(h)
        try:
            if case["kind"] == "dbscan":
                return _run_dbscan(r, case["n"], case["min_pts"])
            if case["kind"] == "knn":
                return _run_knn(r, case["n"], case["k"])
            return _run_pairs(r, case["n"], state["capacity"])
        finally:
            binding.sj_result_free(r)
    finally:
        binding.sj_destroy(h)


def work(case):
    """Each point read once, each result written once; the distance of each
    result pair (each pair at all without an index), a subtraction, a product
    and a sum a dimension."""
    if case["kind"] == "batch":
        nd = [(n, d) for _, n, d in _batch_sizes(case)]
        return {"bytes": sum(8.0 * n * d + 8.0 * 33 * n for n, d in nd), "flops": sum(3.0 * 33 * n * d / 2 for n, d in nd)}
    n, d = case["n"], case["d"]
    pairs = n * (_neighbours(case) + 1.0)
    if case["kind"] == "dbscan":
        out = 4.0 * n
    elif case["kind"] == "knn":
        out = n * (12.0 * case["k"] + 4.0)
    else:
        out = float(n) * n if n <= ADJACENCY else pairs * 8.0
    evaluated = n * (n - 1.0) / 2 if not case.get("index", True) else pairs / 2
    return {"bytes": 8.0 * n * d + out, "flops": 3.0 * d * evaluated}


def exact(case, seed):
    """Distances by brute force in 64 bits (pairs, indices and labels are whole numbers: no value)."""
    if case["kind"] != "knn":
        return None
    x, eps = _points(case, seed)
    n, k, got, rows = case["n"], case["k"], [], max(1, 400_000_000 // case["n"])
    for r0 in range(0, n, rows):
        r1 = min(n, r0 + rows)
        s = torch.zeros((r1 - r0, n), dtype=torch.float64, device=DEV)
        for c in range(case["d"]):
            t = x[r0:r1, c, None] - x[None, :, c]
            s += t * t
        s[s > eps * eps] = math.inf
        s[torch.arange(r1 - r0, device=DEV), torch.arange(r0, r1, device=DEV)] = math.inf
        got.append(torch.topk(s, min(k, n), dim=1, largest=False, sorted=True).values.sqrt())
    return {"idx": None, "dist": torch.cat(got), "found": None}
