"""The neighbour runs of grids of four and more indexed dims (a warp a cell), in
fixed slots (small key spaces) and counted first (large ones), symmetric and
not, with cells at every border of the grid, crowded and single cells: candidate
and evaluation counts of the closed forms, and the oracle's pair set."""
import numpy as np
import pytest

import oracle
from paper_2209_11287_gb300 import binding

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("symmetric", [True, False])
@pytest.mark.parametrize("kernel", ["filter_f32", "fp64_fma"])
@pytest.mark.parametrize("d,m,cells", [(4, 4, 3), (4, 4, 12), (5, 5, 6), (6, 6, 4), (6, 6, 9), (7, 5, 8), (4, 4, 40)])
def test_runs_of_many_offsets(kernel, d, m, cells, symmetric):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = np.random.Generator(np.random.PCG64(cells * 10 + d))
    n = 2500
    x = g.random((n, d))
    x[: n // 4] = np.round(x[: n // 4])  # corners of the grid, crowded
    x[0], x[1] = 0.0, 1.0
    eps = 1.0 / (cells - 0.5)
    ref = oracle.join(x, eps)
    pairs, _, st = binding.self_join(torch.from_numpy(x).cuda(), eps, kernel=kernel, symmetric=symmetric,
                                     indexed_dims=m)
    assert np.array_equal(binding.pairs_to_keys(pairs), ref)
    assert st["m"] == m
    w = eps * (1.0 + 2.0 ** -20)
    cell = np.floor((x[:, :m] - x[:, :m].min(0)) / w).astype(np.int64)  # (all dims have as many cells: the first m)
    uniq, cnt = np.unique(cell, axis=0, return_counts=True)
    near = (np.abs(uniq[:, None, :] - uniq[None, :, :]).max(-1) <= 1) if uniq.shape[0] < 4000 else None
    assert st["n_cells"] == uniq.shape[0]
    assert st["n_candidates"] == int((near * cnt[None, :] * cnt[:, None]).sum())


@pytest.mark.parametrize("symmetric", [True, False])
@pytest.mark.parametrize("kernel", ["filter_f32", "fp64_fma"])
@pytest.mark.parametrize("d,m,cells", [(1, 1, 5_000_000), (2, 2, 2200), (3, 3, 170), (4, 4, 47), (5, 5, 23), (6, 6, 14)])
def test_runs_of_a_sparse_key_space(kernel, d, m, cells, symmetric):
    """Key spaces too large for the counting sort (more than 2^22 keys): cells
    found by search, one pass."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = np.random.Generator(np.random.PCG64(cells + d))
    n = 2500
    eps = 1.0 / (cells - 0.5)
    x = g.random((n, d))
    x[: n // 4] = np.round(x[: n // 4])  # corners of the grid, crowded
    x[n // 2:] = x[n // 4: n // 4 + n - n // 2] + eps * (g.random((n - n // 2, d)) - 0.5)  # neighbours of others
    x = np.clip(x, 0.0, 1.0)
    x[0], x[1] = 0.0, 1.0
    ref = oracle.join(x, eps)
    pairs, _, st = binding.self_join(torch.from_numpy(x).cuda(), eps, kernel=kernel, symmetric=symmetric,
                                     indexed_dims=m)
    assert np.array_equal(binding.pairs_to_keys(pairs), ref)
    assert st["m"] == m
    w = eps * (1.0 + 2.0 ** -20)
    uniq, cnt = np.unique(np.floor((x - x.min(0)) / w).astype(np.int64), axis=0, return_counts=True)
    near = np.abs(uniq[:, None, :] - uniq[None, :, :]).max(-1) <= 1
    assert st["n_cells"] == uniq.shape[0]
    assert st["n_candidates"] == int((near * cnt[None, :] * cnt[:, None]).sum())
