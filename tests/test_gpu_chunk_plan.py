"""Planning of gradients whose tape does not fit one chunk, with few long pairs (the adjoint of such a batch
runs as a strip chain): the chunk is measured against the pairs that are resident with a warp each, so
a batch of at most twice as many pairs as a chunk holds is accepted.  Sizes only; nothing is allocated
or run (the tape of one of these pairs takes 5.4 GB).
"""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu
sk = pytest.importorskip("paper_2502_08470_gb300.sigkernel")


def _size(op, na, nb, n, points, scheme, N, flags=0):
    lib = sk.load_library()
    paths = [sk._Paths(0x10000 * k, 0x10000 * k + 0x1000, c, points, c * points) for k, c in ((1, na), (3, nb))]
    opt = sk._options(scheme, N, 0, "f32", flags)
    size = ctypes.c_size_t(0)
    rc = lib.sigkernel_workspace_size(op, ctypes.byref(paths[0]), ctypes.byref(paths[1]), 4, ctypes.c_int64(n),
                                      ctypes.byref(opt), ctypes.byref(size))
    return rc, size.value


@pytest.mark.parametrize("scheme,N", [("interp", 8), ("approx", 12)])
def test_chunks_of_few_long_pairs(scheme, N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    chunk = 64 << 30  # bytes of tape a chunk may take
    rc, one = _size(sk.OP_BACKWARD, 1, 1, -1, 8193, scheme, N)
    assert rc == 0 and chunk // 16 < one  # 16 pairs do not fit a chunk
    rc, got = _size(sk.OP_BACKWARD, 4, 4, -1, 8193, scheme, N)  # 16 pairs
    # from tapes: more than the checkpointing adjoint, which keeps none, would take
    assert rc == 0 and got > chunk // 2
    rc, got = _size(sk.OP_MMD2, 4, 4, 1, 8193, scheme, N)
    assert rc == 0 and got > chunk // 2
    rc, got = _size(sk.OP_MMD2, 4, 4, 1, 8193, scheme, N, sk.FLAG_UNBIASED)
    assert rc == 0 and got > chunk // 2
