"""The forest of sj_dbscan where its passes differ: long chains in shuffled
order (deep trees; few pairs a point: one hooking round over all pairs), dense
groups (many pairs a point: rounds on a share of them), every point core, no
point core, sizes around the words of the core bit set.  Labels equal the
oracle's exactly."""
import numpy as np
import pytest

import oracle
from paper_2209_11287_gb300 import binding

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _points(kind, n, g):
    if kind == "chain":  # two interleaved chains, neighbours at distance 1
        x = np.stack([np.arange(n) // 2, 5.0 * (np.arange(n) % 2)], axis=1).astype(np.float64)
        return x, 1.0
    if kind == "dense":  # groups of about 80 within eps of each other, bridged by single points
        c = g.integers(0, max(1, n // 80), size=n).astype(np.float64)
        return np.stack([3.0 * c + g.random(n), g.random(n)], axis=1), 1.5
    return 100.0 * np.stack([np.arange(n) % 50, np.arange(n) // 50], axis=1).astype(np.float64), 1.0  # apart


@pytest.mark.parametrize("kind,n,min_pts", [
    ("chain", 20001, 2), ("chain", 20001, 3), ("chain", 33, 3), ("dense", 6000, 1), ("dense", 6000, 40),
    ("dense", 6001, 75), ("dense", 64, 30), ("dense", 31, 1000), ("apart", 65, 1), ("apart", 65, 2)])
def test_forest_matches_oracle(kind, n, min_pts):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = np.random.Generator(np.random.PCG64(n + min_pts))
    x, eps = _points(kind, n, g)
    x = np.ascontiguousarray(x[g.permutation(n)])
    r = binding.sj_join(torch.from_numpy(x).cuda(), eps)
    try:
        labels, k = binding.sj_dbscan(r, n, min_pts)
    finally:
        binding.sj_result_free(r)
    ref, kref = oracle.dbscan(x, eps, min_pts)
    assert k == kref
    assert np.array_equal(labels, ref)
