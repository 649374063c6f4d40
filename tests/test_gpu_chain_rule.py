"""Which batches of FP64 pairs of one length run as a strip chain, by the workspace they are planned with (a
chain's buffers show as the difference to the least workspace; nothing is allocated or run): those
whose blocks of four warps leave an SM with one more than the mean, not those that fill every SM evenly
(once, up to 513 points: beyond, the gaps that a single block leaves cost as much as a chain's fill)."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu
sk = pytest.importorskip("paper_2502_08470_gb300.sigkernel")


def _chained(n, points, N):
    lib = sk.load_library()
    p = sk._Paths(0x10000, 0x1000, n, points, n * points)
    opt = sk._options("approx", N, 0, "f64", 0)
    size = [ctypes.c_size_t(0), ctypes.c_size_t(0)]
    for f, v in zip((lib.sigkernel_workspace_size, lib.sigkernel_workspace_least), size):
        sk._check(f(sk.OP_PAIRS, ctypes.byref(p), ctypes.byref(p), 3, ctypes.c_int64(n), ctypes.byref(opt), ctypes.byref(v)))
    return size[0].value > size[1].value


@pytest.mark.parametrize("points", [257, 513, 1025])
@pytest.mark.parametrize("N", [3, 6])
def test_chain_where_blocks_do_not_spread_evenly(points, N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    slots = 4 * sms  # one block of four warps on each SM
    assert _chained(slots // 4, points, N)
    if points <= 513:
        assert not _chained(slots, points, N)
    assert _chained(slots + 32, points, N)  # a second block on some SMs
    assert not _chained(2 * slots, points, N)
