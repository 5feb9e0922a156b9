"""sj_result_copy of batched results into device memory, whose scattered pages
one kernel gathers: instances of few and of many pages (more than one kernel's
list), a last page of one pair, an unaligned destination (copied page by page),
against the copy into host memory."""
import ctypes

import numpy as np
import pytest

from paper_2209_11287_gb300 import binding

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("page_pairs", [64, 256, 4096])
@pytest.mark.parametrize("emit", [False, True], ids=["pairs", "distances"])
def test_pages_gathered_on_the_device(page_pairs, emit):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = np.random.Generator(np.random.PCG64(21))
    xs = [g.random((n, 2)) for n in (3000, 1, 700, 3500, 65)]
    opt = binding.sj_default_options(page_pairs=page_pairs, emit_distances=int(emit))
    res = binding.sj_join_batch([torch.from_numpy(x).cuda() for x in xs], [0.05] * len(xs), opt)
    try:
        assert max(r.n_pages for r in res) > 448 or page_pairs > 64
        for r in res:
            hp, hd = binding.sj_result_copy(r)
            dp = torch.full((r.count + 3, 2), -7, dtype=torch.int32, device="cuda")
            dd = torch.full((r.count + 3,), -7.0, dtype=torch.float64, device="cuda")
            binding.sj_result_copy(r, dp, dd if emit else None)
            assert np.array_equal(dp.cpu().numpy()[:r.count], hp) and (dp[r.count:] == -7).all()
            if emit:
                assert np.array_equal(dd.cpu().numpy()[:r.count], hd) and (dd[r.count:] == -7.0).all()
            # a destination of 4-byte alignment only
            raw = torch.full((2 * r.count + 2,), -7, dtype=torch.int32, device="cuda")
            assert binding.load().sj_result_copy(ctypes.byref(r), raw.data_ptr() + 4, None) == 0
            assert np.array_equal(raw.cpu().numpy()[1:-1].reshape(-1, 2), hp) and raw[0] == -7 and raw[-1] == -7
    finally:
        for r in res:
            binding.sj_result_free(r)
