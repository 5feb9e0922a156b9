"""Records past the queue of the tensor-core filter are decided and written by
the tile kernel itself, a warp's records together: items of few queries with
half of their columns in (up to a record per candidate and item) and the least
queue (the larger one's allocation fails, injected on the host), uncertain
columns among them, symmetric and not, single and batched, with and without
distances.  Pair sets and distances equal the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2209_11287_gb300 import binding

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _same(x, eps, pairs, dist):
    ref, rd = oracle.join(x, eps, with_dist=True)
    key = (pairs[:, 0].astype(np.int64) << 32) | pairs[:, 1]
    order = np.argsort(key)
    assert np.array_equal(key[order], ref)
    if dist is not None:
        assert np.array_equal(dist[order], rd)


def _with_the_least_queue(run):
    """run() with the one allocation failed that it survives."""
    for k in range(400):
        binding.sj_debug_fail_some_allocations(k, 1)
        try:
            out = run()
        except binding.SimJoinError as e:
            assert e.status == binding.SJ_ERR_OOM
            continue
        finally:
            due = binding.sj_debug_fail_some_allocations(0, 0)
        assert due == 0, "no allocation has a smaller form to fall back on"
        return out


def _points(n, d, seed):
    g = np.random.Generator(np.random.PCG64(seed))
    x = g.random((n, d))
    x[: n // 3] = g.integers(0, 5, (n // 3, d)) / 4.0  # many pairs at equal distances
    return x, float(np.sqrt(d / 6.0))  # about half of the pairs


@pytest.mark.parametrize("emit", [False, True], ids=["pairs", "distances"])
@pytest.mark.parametrize("symmetric", [True, False])
@pytest.mark.parametrize("d,kernel", [(2, "filter_fp16x2"), (16, "filter_bf16x3")])
@pytest.mark.parametrize("qpi", [1, 5, 8])
def test_single(qpi, d, kernel, symmetric, emit):
    x, eps = _points(4001, d, qpi)
    pts = torch.from_numpy(x).cuda()
    pairs, dist, _ = _with_the_least_queue(lambda: binding.self_join(
        pts, eps, kernel=kernel, queries_per_item=qpi, symmetric=symmetric, emit_distances=emit, indexed_dims=-1,
        max_pairs_hint=1 << 24))
    _same(x, eps, pairs, dist)


@pytest.mark.parametrize("emit", [False, True], ids=["pairs", "distances"])
def test_batch(emit):
    sets = [_points(n, 3, k) for k, n in enumerate((2500, 1, 3003, 40, 2002))]
    pts = [torch.from_numpy(x).cuda() for x, _ in sets]
    out = _with_the_least_queue(lambda: binding.join_batch(
        pts, [e for _, e in sets], kernel="filter_fp16x2", queries_per_item=2, indexed_dims=-1, emit_distances=emit))
    for (x, eps), (pairs, dist, _) in zip(sets, out):
        _same(x, eps, pairs, dist)
