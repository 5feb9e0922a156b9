"""The bounding-box prune in front of the FP64 tile and of the FP32 tile with
distances (padded d <= 8): chunk and ring remainders, duplicates, points at
exactly eps, coordinates whose binary32 roundings dwarf eps (a tight cluster far
from the extent's centre), extents that binary32 cannot hold.  Pairs and
distances equal the oracle's exactly."""
import numpy as np
import pytest

import oracle
from paper_2209_11287_gb300 import binding

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _set(kind, d, g):
    if kind == "uniform":
        return g.random((3001, d)), 0.3 if d > 4 else 0.08
    if kind == "lattice":
        return g.integers(0, 9 if d > 2 else 40, size=(2500, d)) / 8.0, 1.0 / 8.0
    if kind == "cancel":  # eps near the binary32 rounding of the coordinates
        x = 1e4 + 1e-3 * g.random((1500, d))
        x[:3] = -1e4
        return x, 2e-4
    scale = {"huge": 1e60, "tiny": 1e-60}[kind]
    return g.random((2000, d)) * scale, (0.3 if d > 4 else 0.08) * scale


@pytest.mark.parametrize("kernel,emit", [("fp64_fma", False), ("fp64_fma", True), ("filter_f32", True)])
@pytest.mark.parametrize("kind", ["uniform", "lattice", "cancel", "huge", "tiny"])
@pytest.mark.parametrize("d", [2, 3, 4, 7, 8])
def test_pruned_tiles(kernel, emit, kind, d):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    x, eps = _set(kind, d, np.random.Generator(np.random.PCG64(d)))
    ref, rd = oracle.join(x, eps, with_dist=True)
    for qpi in (0, 3):
        pairs, dist, _ = binding.self_join(torch.from_numpy(x).cuda(), eps, kernel=kernel, emit_distances=emit,
                                           queries_per_item=qpi)
        key = (pairs[:, 0].astype(np.int64) << 32) | pairs[:, 1]
        order = np.argsort(key)
        assert np.array_equal(key[order], ref)
        if emit:
            assert np.array_equal(dist[order], rd)
