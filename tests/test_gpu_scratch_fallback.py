"""Scratch that makes do with less when memory is short: one allocation (or two
in a row) of a call fails and those after it succeed (injected on the host).
Each attempt either ends with SJ_ERR_OOM and nothing kept, or returns the
oracle's result with no error message left behind; the ones that have a smaller
form to fall back on must succeed."""
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
    yield
    binding.sj_debug_fail_some_allocations(0, 0)


def _sweep(run, check, count=1):
    """Fails the allocations k .. k + count - 1 of the call for k = 0, 1, ...
    up to its last one: those it survived."""
    check(run()[0])
    torch.cuda.synchronize()
    base = binding.sj_debug_live_allocations()
    survived = []
    for k in range(400):
        binding.sj_debug_fail_some_allocations(k, count)
        try:
            out, message = run()
        except binding.SimJoinError as e:
            assert e.status == binding.SJ_ERR_OOM, (k, e)
            out = None
        finally:
            due = binding.sj_debug_fail_some_allocations(0, 0)
        torch.cuda.synchronize()
        assert binding.sj_debug_live_allocations() == base, k
        if out is not None:
            check(out)
            if due > 0:
                return survived
            assert message == "", (k, message)
            survived.append(k)
    raise AssertionError("the call never ran to its end")


def _join(pts, eps, **opt):
    r = binding.sj_join(pts, eps, binding.sj_default_options(**opt))
    message = binding.sj_last_error_message()
    out = binding.sj_result_copy(r)
    binding.sj_result_free(r)
    return out, message


def _points(n, seed):
    g = np.random.Generator(np.random.PCG64(seed))
    return g.random((n, 2))


def _keys(pairs):
    return binding.pairs_to_keys(pairs)


@pytest.mark.parametrize("emit", [False, True], ids=["pairs", "distances"])
def test_record_queue_of_one_join(emit):
    x, eps = _points(5001, 1), 0.04
    ref, rd = oracle.join(x, eps, with_dist=True)
    pts = torch.from_numpy(x).cuda()

    def check(out):
        key = (out[0][:, 0].astype(np.int64) << 32) | out[0][:, 1]
        order = np.argsort(key)
        assert np.array_equal(key[order], ref)
        if emit:
            assert np.array_equal(out[1][order], rd)

    # no index, one query an item: more than 2^23 evaluations, so the queue asks for more than its least size
    survived = _sweep(lambda: _join(pts, eps, kernel="filter_fp16x2", indexed_dims=-1, queries_per_item=1,
                                    emit_distances=int(emit), max_pairs_hint=1 << 20), check)
    assert emit or len(survived) == 1


def test_record_queue_of_a_join_to_host():
    x, eps = _points(5001, 2), 0.04
    ref = oracle.join(x, eps)
    pts = torch.from_numpy(x).cuda()

    def run():
        h = binding.sj_build_index(pts, eps, binding.sj_default_options(kernel="filter_fp16x2", indexed_dims=-1,
                                                                        queries_per_item=1))
        try:
            out = np.empty((ref.size, 2), dtype=np.int32)
            cnt, _ = binding.sj_self_join_to_host(h, out, 1 << 20)
            return out[:cnt], binding.sj_last_error_message()
        finally:
            binding.sj_destroy(h)

    assert len(_sweep(run, lambda out: np.testing.assert_array_equal(_keys(out), ref))) == 1


def test_record_queues_of_a_batch():
    # two tensor groups: where not even the least queue of the second fits
    # beside the first one's, both are taken at their least size
    g = np.random.Generator(np.random.PCG64(3))
    sets = [(g.random((5001, 2)), 0.04), (g.random((5001, 9)), 0.3)]
    refs = [oracle.join(x, e) for x, e in sets]
    pts = [torch.from_numpy(x).cuda() for x, _ in sets]

    def run():
        res = binding.sj_join_batch(pts, [e for _, e in sets], binding.sj_default_options(
            kernel="filter_fp16x2", indexed_dims=-1, queries_per_item=1, max_pairs_hint=1 << 22))
        message = binding.sj_last_error_message()
        out = [binding.sj_result_copy(r)[0] for r in res]
        for r in res:
            binding.sj_result_free(r)
        return out, message

    def check(out):
        for p, ref in zip(out, refs):
            assert np.array_equal(_keys(p), ref)

    assert len(_sweep(run, check)) >= 2
    assert len(_sweep(run, check, count=2)) >= 1


def test_runs_of_a_sparse_key_space():
    """The runs in fixed slots and the items beside them: packed runs instead."""
    g = np.random.Generator(np.random.PCG64(4))
    x, eps = g.random((6000, 3)), 0.004
    ref = oracle.join(x, eps)
    pts = torch.from_numpy(x).cuda()
    infos = []

    def run():
        h = binding.sj_build_index(pts, eps, binding.sj_default_options(kernel="filter_f32"))
        message = binding.sj_last_error_message()
        due = binding.sj_debug_fail_some_allocations(0, 0)  # (the build's allocations only)
        r = binding.sj_self_join(h)
        out = binding.sj_result_copy(r)[0]
        infos.append(binding.sj_index_info(h))
        binding.sj_result_free(r)
        binding.sj_destroy(h)
        binding.sj_debug_fail_some_allocations(1 << 30, due)
        return out, message

    assert len(_sweep(run, lambda out: np.testing.assert_array_equal(_keys(out), ref))) >= 2
    assert all(i == infos[0] for i in infos)


def test_list_of_the_items_of_many_queries():
    """Crowded cells among single points: without the list that the two FP32
    filters share the items by, one of them takes all."""
    g = np.random.Generator(np.random.PCG64(5))
    n = 260_000
    x = g.random((n, 3))
    eps = (0.3 / n) ** (1.0 / 3)
    x[: n // 4] = x[g.integers(n // 2, n // 2 + 4000, n // 4)] + 0.05 * eps * g.random((n // 4, 3))
    ref = oracle.join(x, eps)
    h = binding.sj_build_index(torch.from_numpy(x).cuda(), eps,
                               binding.sj_default_options(kernel="filter_f32", max_pairs_hint=1 << 24))

    def run():
        launches = binding.sj_kernel_launches()
        r = binding.sj_self_join(h)
        message = binding.sj_last_error_message()
        kernels.append(binding.sj_kernel_launches() - launches)
        out = binding.sj_result_copy(r)[0]
        binding.sj_result_free(r)
        return out, message

    kernels = []
    try:
        survived = _sweep(run, lambda out: np.testing.assert_array_equal(_keys(out), ref))
    finally:
        binding.sj_destroy(h)
    assert len(survived) == 1
    assert kernels[0] == kernels[1] + 1 == kernels[2]  # (two tile kernels where the list is there)


@pytest.mark.parametrize("k", [4, 30, 200])
def test_entries_of_the_knn_selection(k):
    """Without room for 16 bytes a pair and its place: 12 bytes a pair."""
    x, eps = _points(3000, 6), 0.12
    r = binding.sj_join(torch.from_numpy(x).cuda(), eps, binding.sj_default_options(emit_distances=1))
    want = binding.sj_knn_from_join(r, x.shape[0], k)

    def run():
        out = binding.sj_knn_from_join(r, x.shape[0], k)
        return out, binding.sj_last_error_message()

    def check(out):
        for a, b in zip(out, want):
            assert np.array_equal(a, b)

    try:
        assert len(_sweep(run, check)) == 2
    finally:
        binding.sj_result_free(r)
