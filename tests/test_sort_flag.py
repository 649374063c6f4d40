"""Which calls of the binding leave out ordering the pairs by their cells: those on sets known to have paths of
one length, not those on a set whose offsets only the device knows, however many rows its buffer has."""
import pytest
import torch

from paper_2502_08470_gb300 import workloads as W

sk = pytest.importorskip("paper_2502_08470_gb300.sigkernel")


def test_flags():
    dense = sk.Paths.from_dense(torch.zeros(3, 5, 2))
    longer = sk.Paths.from_dense(torch.zeros(2, 6, 2))
    equal = sk.Paths.from_list([torch.zeros(5, 2)] * 4, device="cpu")
    ragged = sk.Paths.from_list([torch.zeros(5, 2), torch.zeros(2, 2)], device="cpu")
    room = sk.Paths(torch.zeros(10, 2), torch.tensor([0, 5, 7]), 5)  # two paths in a buffer for two of 5 rows
    no = sk.FLAG_NO_SORT
    for X, Y, flag in [(dense, dense, no), (dense, longer, no), (dense, equal, no), (dense, ragged, 0), (ragged, dense, 0),
                       (room, dense, 0), (room, room, 0)]:
        assert sk._sort_flag(True, X, Y) == flag
        assert sk._sort_flag(False, X, Y) == no


@pytest.mark.gpu
def test_ragged_set_in_a_buffer_with_room_is_sorted():
    """FD pairs in the pipeline, a short one first: taken in the given order its block, and every other one, falls
    back to a warp per pair."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lens = [3] * 152 + [1500] * 40
    rows = torch.as_tensor(W.brownian(1, sum(lens), 2, seed=781)[0], dtype=torch.float32, device="cuda")
    off = torch.tensor([0] + lens, dtype=torch.int64).cumsum(0).to("cuda")
    buffer = torch.zeros(len(lens) * 1500, 2, device="cuda")
    buffer[:len(rows)] = rows
    X = sk.Paths(buffer, off, 1500)
    i = torch.arange(len(lens), device="cuda")
    ms, out = {}, {}
    for sort in (True, False):
        for _ in range(2):
            out[sort] = sk.sigkernel_pairs(X, X, i, i, scheme="fd1", degree=0, compute="f32", sort=sort, strip_pipeline=True,
                                           time_kernel=True)
        ms[sort] = sk.last_kernel_ms()
    assert sk.device_status() == 0
    assert torch.equal(out[True], out[False])
    assert ms[True] < 0.6 * ms[False]  # 47 strips: by 16 warps together, or by one after another
