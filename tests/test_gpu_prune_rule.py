"""Joins on both sides of the line from which candidates pass the bounding-box
prune (140 candidates an item, 70 in the plane, 90 for few items in FP64): the
FP32 tile with distances performs fewer evaluations than scheduled above it and
every one below it and without an index; pairs and distances of both tiles equal the
oracle's on either side."""
import numpy as np
import pytest

import oracle
from paper_2209_11287_gb300 import binding

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("kernel,emit", [("fp64_fma", False), ("fp64_fma", True), ("filter_f32", True)])
@pytest.mark.parametrize("d,share,indexed", [(2, 30, 0), (2, 69, 0), (2, 72, 0), (2, 300, 0), (3, 80, 0), (3, 100, 0), (3, 128, 0), (3, 139, 0),
                                             (3, 141, 0), (3, 400, 0), (4, 60, 0), (4, 170, 0), (5, 300, 0),
                                             (8, 900, 0), (3, 300, -1)])
def test_both_sides(d, share, indexed, kernel, emit):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = 6000
    g = np.random.Generator(np.random.PCG64(d * 1000 + share))
    x = g.random((n, d))
    # cells of side eps: share = n (half of the 3^d cells of a neighbourhood) eps^d, away from the edges
    eps = float((2 * share / (n * 3.0 ** d)) ** (1.0 / d))
    ref, rd = oracle.join(x, eps, with_dist=True)
    pairs, dist, st = binding.self_join(torch.from_numpy(x).cuda(), eps, kernel=kernel, emit_distances=emit,
                                        indexed_dims=indexed)
    key = (pairs[:, 0].astype(np.int64) << 32) | pairs[:, 1]
    order = np.argsort(key)
    assert np.array_equal(key[order], ref)
    if emit:
        assert np.array_equal(dist[order], rd)
    if kernel == "filter_f32":
        prune = indexed == 0 and st["n_evaluated"] > (140 if d > 2 else 70) * n
        assert (st["n_performed"] < st["n_evaluated"]) == prune
