"""The tensor-core filter's records and their resolution (k_resolve) where they
can go wrong: more records than the queue holds (one query per item and a
bound that certifies nothing: a record per evaluated pair), items of few and of
many query columns, a tile with a 16-column tail, runs cut into many copies,
batched joins whose warps meet several instances, with and without distances.
Pair sets and distances equal the oracle's exactly."""
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


def _check(x, eps, emit, **opt):
    ref, rd = oracle.join(x, eps, with_dist=True)
    pairs, dist, st = binding.self_join(torch.from_numpy(x).cuda(), eps, emit_distances=emit, **opt)
    key = (pairs[:, 0].astype(np.int64) << 32) | pairs[:, 1]
    order = np.argsort(key)
    assert np.array_equal(key[order], ref)
    if emit:
        assert np.array_equal(dist[order], rd)
    return st


@pytest.mark.parametrize("emit", [False, True], ids=["pairs", "distances"])
def test_more_records_than_the_queue_holds(emit):
    g = np.random.Generator(np.random.PCG64(8))
    # one far point: no pair is certified by the tile's bound
    x = np.concatenate([g.random((12000, 2)), [[1.0e4, 1.0e4]]])
    st = _check(x, 0.05, emit, kernel="filter_fp16x2", queries_per_item=1)
    assert st["n_rechecked"] > (1 << 19)  # (2^19 records fit)


@pytest.mark.parametrize("kernel", ["filter_fp16x2", "filter_bf16x2", "filter_bf16x3"])
@pytest.mark.parametrize("d,n,qpi", [(2, 3000, 0), (3, 5000, 5), (8, 3000, 17), (16, 2500, 33), (16, 3001, 0),
                                     (33, 1500, 0), (64, 1200, 0), (64, 900, 100)])
def test_shapes(kernel, d, n, qpi):
    g = np.random.Generator(np.random.PCG64(d * 1000 + n))
    c = g.random((6, d))
    x = c[g.integers(0, 6, n)] + 0.05 * g.standard_normal((n, d))
    # about 30 neighbours
    s = np.sort(((x[:60, None, :] - x[None, :, :]) ** 2).sum(-1), axis=1)[:, 30]
    _check(x, float(np.sqrt(np.median(s))), False, kernel=kernel, queries_per_item=qpi)


@pytest.mark.parametrize("emit", [False, True], ids=["pairs", "distances"])
def test_batch_of_small_instances(emit):
    g = np.random.Generator(np.random.PCG64(3))
    xs = [g.random((int(m), 8)) * 10.0 ** (k % 7 - 3) for k, m in enumerate(g.integers(1, 90, 200))]
    eps = [0.45 * 10.0 ** (k % 7 - 3) for k in range(len(xs))]
    out = binding.join_batch([torch.from_numpy(x).cuda() for x in xs], eps, kernel="filter_fp16x2",
                             emit_distances=emit)
    for x, e, (pairs, dist, _) in zip(xs, eps, out):
        ref, rd = oracle.join(x, e, with_dist=True)
        key = (pairs[:, 0].astype(np.int64) << 32) | pairs[:, 1]
        order = np.argsort(key)
        assert np.array_equal(key[order], ref)
        if emit:
            assert np.array_equal(dist[order], rd)


def test_batch_of_many_records():
    """Enough of them that a warp takes several blocks of records in a row,
    over the edges of instances."""
    g = np.random.Generator(np.random.PCG64(4))
    xs = [g.random((int(m), 2)) for m in g.integers(100, 1800, 48)]
    eps = [float(np.sqrt(120 / (np.pi * len(x)))) for x in xs]
    out = binding.join_batch([torch.from_numpy(x).cuda() for x in xs], eps, kernel="filter_fp16x2",
                             queries_per_item=1)
    for x, e, (pairs, _, _) in zip(xs, eps, out):
        ref, _ = oracle.join(x, e, with_dist=True)
        assert np.array_equal(np.sort((pairs[:, 0].astype(np.int64) << 32) | pairs[:, 1]), ref)
