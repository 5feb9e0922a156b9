"""The kNN selection on both sides of the line from which its entries are split
into indices and distances (3 * 2^22 pairs of at least 128 neighbours a point): the
neighbours and distances of every point equal those that its row of the pairs,
sorted by (distance, index), begins with."""
import numpy as np
import pytest

from paper_2209_11287_gb300 import binding

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,side,k", [(3547, 9.0, 5), (3548, 9.0, 5), (3600, 9.0, 300), (20000, 160.0, 20)])
def test_both_forms(n, side, k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = np.random.Generator(np.random.PCG64(n))
    x = torch.from_numpy(g.integers(0, 64, (n, 2)) * (side / 64.0)).cuda()  # (equal distances among them)
    r = binding.sj_join(x, 13.0, binding.sj_default_options(emit_distances=1))
    try:
        idx, dist, found = binding.sj_knn_from_join(r, n, k)
        pairs, pd = binding.sj_result_copy(r)
    finally:
        binding.sj_result_free(r)
    if side < 13.0 / np.sqrt(2):
        assert pairs.shape[0] == n * n  # everything is a neighbour: 3 * 2^22 lies between the first two sizes
    keep = pairs[:, 0] != pairs[:, 1]
    i, j, d = pairs[keep, 0], pairs[keep, 1], pd[keep]
    order = np.lexsort((j, d, i))
    i, j, d = i[order], j[order], d[order]
    start = np.searchsorted(i, np.arange(n + 1))
    size = np.minimum(np.diff(start), k)
    assert np.array_equal(found, size)
    at = start[:-1, None] + np.arange(k)[None, :]
    inside = np.arange(k)[None, :] < size[:, None]
    at = np.minimum(at, j.size - 1)
    assert np.array_equal(idx, np.where(inside, j[at], -1))
    assert np.array_equal(dist, np.where(inside, d[at], np.inf))
