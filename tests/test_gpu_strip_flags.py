"""SK_FLAG_STRIP_PIPELINE and SK_FLAG_NO_STRIP_PIPELINE in the forward that records a tape and in its adjoint:
with the second, one warp per pair (a limit of one poll, which the waits of a chain of few pairs exhaust,
then changes nothing, and the workspace has no hand-off buffers); with the first, a chain also where the
library would not choose one (10000 pairs, whose first strips are all done before a second one starts:
nothing waits, and only the workspace shows the chain).  The values are the same.
"""
import ctypes

import pytest
import torch

from paper_2502_08470_gb300 import workloads as W

pytestmark = pytest.mark.gpu
sk = pytest.importorskip("paper_2502_08470_gb300.sigkernel")

SK_ERR_DEVICE_TIMEOUT = -5


def _run(X, flags, limit, scheme, N):
    """Values, gradients, device status and workspace size of a tape forward and its adjoint."""
    lib = sk.load_library()
    X = sk.as_paths(X)
    c, n = sk._cpaths(X), X.count
    opt = sk._options(scheme, N, 0, "f32", flags | sk.FLAG_NO_TC)
    nb = ctypes.c_size_t(0)
    ref = ctypes.byref
    sk._check(lib.sigkernel_tape_size(ref(c), ref(c), X.d, ctypes.c_int64(-1), ref(opt), ref(nb)))
    tape = torch.empty(nb.value, dtype=torch.uint8, device="cuda")
    ws = sk._workspace(sk.OP_GRAM, c, c, X.d, -1, opt)
    wb = sk._workspace(sk.OP_BACKWARD_TAPE, c, c, X.d, -1, opt)
    K = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    g = torch.zeros(X.rows.shape, dtype=torch.float64, device="cuda")
    w = torch.ones(n, n, dtype=torch.float64, device="cuda")
    st = torch.cuda.current_stream().cuda_stream
    status = []
    sk.set_wait_limit(limit)
    try:
        sk._check(lib.sigkernel_forward_tape(ref(c), ref(c), X.d, 1, None, None, ctypes.c_int64(-1), ref(opt), K.data_ptr(),
                                             tape.data_ptr(), nb.value, ws.data_ptr(), ws.numel(), st))
        status.append(sk.device_status())
        sk._check(lib.sigkernel_backward_tape(ref(c), ref(c), X.d, 1, None, None, ctypes.c_int64(-1), ref(opt), tape.data_ptr(),
                                              nb.value, w.data_ptr(), g.data_ptr(), None, wb.data_ptr(), wb.numel(), st))
        status.append(sk.device_status())
    finally:
        sk.set_wait_limit(0)
    return K, g, status, ws.numel()


@pytest.mark.parametrize("scheme,N", [("approx", 4), ("interp", 4)])
@pytest.mark.parametrize("n,points,chosen", [(3, 200, True), (100, 40, False)])
def test_flags_reach_the_tape(scheme, N, n, points, chosen):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    X = torch.as_tensor(W.brownian(n, points, 3, seed=731), dtype=torch.float32, device="cuda")
    assert sk.device_status() == 0
    K0, g0, status, small = _run(X, sk.FLAG_NO_STRIP_PIPELINE, 1, scheme, N)
    assert status == [0, 0]
    waits = [SK_ERR_DEVICE_TIMEOUT] * 2 if chosen else [0, 0]
    *_, status, large = _run(X, sk.FLAG_STRIP_PIPELINE, 1, scheme, N)
    assert status == waits and large > small
    *_, status, size = _run(X, 0, 1, scheme, N)
    assert status == waits and size == (large if chosen else small)
    K1, g1, status, _ = _run(X, sk.FLAG_STRIP_PIPELINE, 0, scheme, N)
    assert status == [0, 0]
    assert torch.equal(K0, K1)
    assert (g0 - g1).abs().max() <= 1e-4 * g0.abs().max()  # FP32 column sums in another order
