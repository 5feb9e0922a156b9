"""The selection of sj_knn_from_join at the sizes where its forms change: a
bucket of neighbours around a multiple of the warp, around the selection's
list of 256 entries and beyond it (the list cut back to its k smallest), and k
around the largest the list is cut back to (early, after the first 32 neighbours, or
when it is full).  Groups of points far apart on an
integer lattice, so many distances of a bucket are equal and the index
decides; the result is the oracle's exactly."""
import numpy as np
import pytest

import oracle
from paper_2209_11287_gb300 import binding

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

GROUPS = (1, 2, 32, 33, 34, 64, 65, 66, 128, 129, 130, 224, 225, 256, 257, 258, 289, 700)


def _groups():
    g = np.random.Generator(np.random.PCG64(5))
    pts = []
    for at, size in enumerate(GROUPS):
        p = g.integers(0, 9, size=(size, 3)).astype(np.float64)
        p[:, 0] += 100.0 * at
        pts.append(p)
    x = np.concatenate(pts)
    return np.ascontiguousarray(x[g.permutation(x.shape[0])])


@pytest.fixture(scope="module")
def joined():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    x, eps = _groups(), 20.0  # every point of a group is a neighbour of the others
    keys, dist = oracle.join(x, eps, with_dist=True)
    i, j = keys >> 32, keys & 0xFFFFFFFF
    order = np.lexsort((j, dist, i))
    i, j, dist = i[order], j[order], dist[order]
    keep = i != j
    r = binding.sj_join(torch.from_numpy(x).cuda(), eps, binding.sj_default_options(emit_distances=1))
    yield x, r, i[keep], j[keep], dist[keep]
    binding.sj_result_free(r)


@pytest.mark.parametrize("k", [1, 16, 24, 25, 33, 192, 193, 256, 300, 1024])
def test_selection_at_its_edges(joined, k):
    x, r, i, j, dist = joined
    n = x.shape[0]
    idx, dd, found = binding.sj_knn_from_join(r, n, k)
    start = np.searchsorted(i, np.arange(n + 1))
    size = np.diff(start)
    assert sorted(set(size + 1)) == sorted(GROUPS)
    assert np.array_equal(found, np.minimum(size, k))
    for p in range(n):
        c = min(size[p], k)
        assert np.array_equal(idx[p, :c], j[start[p]:start[p] + c])
        assert np.array_equal(dd[p, :c], dist[start[p]:start[p] + c])
        assert (idx[p, c:] == -1).all() and np.isinf(dd[p, c:]).all()
