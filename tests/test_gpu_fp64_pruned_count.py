"""The evaluations that the bounding-box prune removes from the FP64 tile are
counted (sj_index_last_pruned), as many as it removes from the FP32 tile with
distances on the same items, and bench.py's FP64 rate counts the others only."""
import json
import os
import subprocess
import sys

import pytest

from paper_2209_11287_gb300 import binding, workloads

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _pruned(w, eps, **opt):
    h = binding.sj_build_index(torch.from_numpy(w.points).cuda(), eps, binding.sj_default_options(**opt))
    try:
        r = binding.sj_self_join(h)
        out = binding.sj_index_last_pruned(h), binding.sj_index_info(h)["n_evaluated"], int(r.n_evaluated)
        binding.sj_result_free(r)
        return out
    finally:
        binding.sj_destroy(h)


def test_counted_for_the_fp64_tile():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    w = workloads.uniform4d(n=40000, seed=21)
    p64, ev, reported = _pruned(w, w.eps, kernel="fp64_fma")
    p32, ev32, _ = _pruned(w, w.eps, kernel="filter_f32", emit_distances=1)
    assert ev == ev32 == reported
    # the radii differ by the bounds of the two coordinate roundings only
    assert p64 == pytest.approx(p32, rel=1e-3) and 0.3 * ev < p64 < 0.65 * ev
    assert _pruned(w, w.eps / 3, kernel="fp64_fma")[0] == 0  # (few candidates an item: not pruned)


def test_bench_counts_what_the_tile_evaluates():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--n", "60000", "--steps", "1", "--warmup",
                        "3", "--no-cpu-baseline", "--variants", "fp64_fma"], capture_output=True, text=True,
                       timeout=300, cwd=ROOT)
    assert r.returncode == 0, r.stderr[-2000:]
    line = json.loads(r.stdout.strip().splitlines()[-1])
    # half of the candidates are scheduled, about half of those evaluated
    assert line["variants"]["fp64_fma"]["evaluated_pairs"] < 0.4 * line["config"]["candidate_pairs"]
