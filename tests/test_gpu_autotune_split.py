"""sigkernel_autotune on FP64 pairs of one strip, where the library shares each pair among four warps by itself:
that shape is among those timed, so the time it returns is that of the calls that follow, and a tuned
call takes the shape that was chosen (another call of the same shape, tuned or not, has the same
values)."""
import pytest
import torch

from paper_2502_08470_gb300 import workloads as W

pytestmark = pytest.mark.gpu
sk = pytest.importorskip("paper_2502_08470_gb300.sigkernel")


def test_shared_pairs_are_among_the_candidates():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    X = sk.as_paths(torch.as_tensor(W.brownian(1, 33, 2, seed=771), dtype=torch.float64, device="cuda"))
    i0 = torch.zeros(1, dtype=torch.int64, device="cuda")
    kw = dict(scheme="approx", degree=4, compute="f64")
    sk.autotune_clear()
    try:
        want = sk.sigkernel_pairs(X, X, i0, i0, **kw)
        sk.sigkernel_pairs(X, X, i0, i0, strip_pipeline=False, time_kernel=True, **kw)  # one warp per pair, asked for
        one = sk.last_kernel_ms()
        sk.sigkernel_pairs(X, X, i0, i0, time_kernel=True, **kw)
        shared = sk.last_kernel_ms()
        assert shared < 0.8 * one  # four warps against one on a chain of FP64 steps
        shape, ms = sk.autotune(X, X, pair_a=i0, pair_b=i0, trials=5, **kw)
        assert shape == {"warps_per_block": 0, "strip_pipeline": False}
        got = sk.sigkernel_pairs(X, X, i0, i0, time_kernel=True, **kw)
        assert sk.last_kernel_ms() < 0.8 * one
        assert torch.equal(got, want)
        # tuned again, with the choice remembered
        assert sk.autotune(X, X, pair_a=i0, pair_b=i0, trials=5, **kw)[0] == shape
        assert sk.device_status() == 0
    finally:
        sk.autotune_clear()
