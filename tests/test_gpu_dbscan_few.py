"""sj_dbscan with few pairs (straight to the pass over all pairs) and on both
sides of that line (six pairs a point, 32768 pairs), down to one point; labels
and cluster counts equal the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2209_11287_gb300 import binding

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("min_pts", [1, 2, 5])
@pytest.mark.parametrize("n,per", [(1, 1), (2, 2), (31, 3), (33, 3), (300, 2), (300, 5.8), (300, 6.4), (5400, 5.7),
                                   (5400, 6.3), (9000, 3), (20000, 2)])
def test_few_pairs(n, per, min_pts):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    x = np.random.Generator(np.random.PCG64(n)).random((n, 2))
    eps = float(np.sqrt(max(per - 1, 0.01) / (np.pi * n)))  # about `per` pairs a point, itself included
    ref, k = oracle.dbscan(x, eps, min_pts)
    r = binding.sj_join(torch.from_numpy(x).cuda(), eps)
    try:
        labels, got = binding.sj_dbscan(r, n, min_pts)
    finally:
        binding.sj_result_free(r)
    assert got == k and np.array_equal(labels, ref)
