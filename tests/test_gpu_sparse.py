"""The FP32 filter for sparse cells (k_join_f32r), alone and beside k_join_f32s: groups of items whose runs
fill the warp's list (27, 81 and 243 runs an item), items of one and of several
queries, uncertain pairs and a recheck queue that overflows nowhere, ranges of
items and rounds to the host, symmetric and not; the oracle's pair set, and the
evaluations of the index (this kernel prunes nothing)."""
import numpy as np
import pytest

import oracle
from paper_2209_11287_gb300 import binding

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _set(kind, n, d, g):
    if kind == "uniform":
        return g.random((n, d)), (0.35 / n) ** (1.0 / d)
    if kind == "lattice":  # many pairs at exactly eps (uncertain), few points a cell
        return g.integers(0, int(2 * n ** (1.0 / d)), size=(n, d)) / 8.0, 1.0 / 8.0
    if kind == "crowded":  # a few crowded cells among single points: both kernels share the items
        x = g.random((n, d))
        x[: n // 3] = 0.5 + 0.02 * (g.random((n // 3, d)) - 0.5) + 0.25 * g.integers(0, 2, (n // 3, 1))
        return x, (0.3 / n) ** (1.0 / d)
    x = g.random((n, d))  # near-duplicates of a few points among single ones
    x[: n // 8] = x[g.integers(n // 8, n // 6, n // 8)] + 1e-9 * g.standard_normal((n // 8, d))
    return x, (0.3 / n) ** (1.0 / d)


@pytest.mark.parametrize("symmetric", [True, False])
@pytest.mark.parametrize("kind", ["uniform", "lattice", "duplicates", "crowded"])
@pytest.mark.parametrize("d", [1, 2, 3, 4, 5, 6, 8])
def test_sparse_cells(d, kind, symmetric):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = np.random.Generator(np.random.PCG64(d))
    x, eps = _set(kind, 7001, d, g)
    ref = oracle.join(x, eps)
    opt = binding.sj_default_options(kernel="filter_f32", symmetric=int(symmetric))
    h = binding.sj_build_index(torch.from_numpy(x).cuda(), eps, opt)
    try:
        info = binding.sj_index_info(h)
        r = binding.sj_self_join(h)
        pairs, _ = binding.sj_result_copy(r)
        assert np.array_equal(binding.pairs_to_keys(pairs), ref)
        if kind == "uniform" and d <= 4:
            assert r.n_evaluated == info["n_evaluated"]
        binding.sj_result_free(r)
        if symmetric:  # shards of whole cells, and rounds
            work = binding.sj_index_item_work(h)
            b = binding.sj_shard_bounds(work, 3)
            got = []
            for k in range(3):
                r = binding.sj_self_join_range(h, b[k], b[k + 1])
                got.append(binding.sj_result_copy(r)[0])
                binding.sj_result_free(r)
            assert np.array_equal(binding.pairs_to_keys(np.concatenate(got)), ref)
            out = np.empty((ref.size, 2), dtype=np.int32)
            cnt, _ = binding.sj_self_join_to_host(h, out, max(1024, ref.size // 4))
            assert cnt == ref.size and np.array_equal(binding.pairs_to_keys(out), ref)
    finally:
        binding.sj_destroy(h)
