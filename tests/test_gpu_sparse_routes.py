"""The FP32 filter for sparse cells where the ordinary sparse sets do not reach:
more uncertain pairs than the recheck queue holds (decided in place), and the
bounds-checking build on the joins that run it alone and beside k_join_f32s
(told apart by the launches of the join)."""
import os
import subprocess
import sys
import textwrap

import numpy as np
import pytest

import oracle
from paper_2209_11287_gb300 import binding

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_more_uncertain_pairs_than_the_queue_holds():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    # a cubic lattice: every neighbour at exactly eps; cells a little wider than
    # that, so the first two layers of each dim share one
    k = 74
    x = np.stack(np.meshgrid(*[np.arange(k) / 8.0] * 3, indexing="ij"), axis=-1).reshape(-1, 3)
    x = np.ascontiguousarray(x[np.random.Generator(np.random.PCG64(1)).permutation(x.shape[0])])
    pairs, _, st = binding.self_join(torch.from_numpy(x).cuda(), 1.0 / 8.0, kernel="filter_f32")
    assert st["n_cells"] == (k - 1) ** 3 and st["n_performed"] == st["n_evaluated"]  # (the kernel that prunes nothing)
    assert st["n_rechecked"] > 1 << 20  # (the queue's size here)
    assert np.array_equal(binding.pairs_to_keys(pairs), oracle.join(x, 1.0 / 8.0))


SCRIPT = textwrap.dedent("""
    import sys
    import numpy as np
    import torch
    sys.path.insert(0, {root!r})
    import oracle
    from paper_2209_11287_gb300 import binding
    g = np.random.Generator(np.random.PCG64(11))
    for d in (2, 3, 4, 6, 8):
        for crowded in (False, True):
            n = 6001 if not crowded else 260_000 if d < 6 else 30_000
            x = g.random((n, d))
            eps = (0.3 / n) ** (1.0 / d)
            if crowded:  # a quarter of the points close to a few others
                x[: n // 4] = x[g.integers(n // 2, n // 2 + n // 64, n // 4)] + 0.05 * eps * g.random((n // 4, d))
            ref = oracle.join(x, eps)
            for sym in (1, 0):
                h = binding.sj_build_index(torch.from_numpy(x).cuda(), eps,
                                           binding.sj_default_options(kernel="filter_f32", symmetric=sym))
                launches = binding.sj_kernel_launches()
                r = binding.sj_self_join(h)
                launches = binding.sj_kernel_launches() - launches
                pairs = binding.sj_result_copy(r)[0]
                assert np.array_equal(binding.pairs_to_keys(pairs), ref), (d, crowded, sym)
                if d in (2, 3, 4):  # tile kernels and the recheck
                    assert launches == (3 if crowded else 2), (d, crowded, sym, launches)
                    assert crowded or r.n_evaluated == binding.sj_index_info(h)["n_evaluated"]
                binding.sj_result_free(r)
                binding.sj_destroy(h)
    print("debug-bounds ok")
""")


def test_debug_bounds_build_passes_every_check_of_the_sparse_filter():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2209_11287_gb300 import build
    env = dict(os.environ, SJ_LIBRARY=build.build(debug_bounds=True))
    r = subprocess.run([sys.executable, "-c", SCRIPT.format(root=ROOT)], env=env, capture_output=True, text=True,
                       timeout=900)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    assert "debug-bounds ok" in r.stdout
