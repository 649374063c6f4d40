"""sigkernel_set_wait_limit in the adjoint of few pairs (a strip chain): with one poll its first hand-off wait
runs out and SK_ERR_DEVICE_TIMEOUT is recorded; the kernel returns, and the next call, from the same tape
with the default limit, has the gradients of the call before."""
import pytest
import torch

from paper_2502_08470_gb300 import workloads as W

pytestmark = pytest.mark.gpu
sk = pytest.importorskip("paper_2502_08470_gb300.sigkernel")

SK_ERR_DEVICE_TIMEOUT = -5


@pytest.mark.parametrize("scheme", ["approx", "interp"])
def test_exhausted_wait_of_the_adjoint(scheme):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    X, Y = (torch.as_tensor(W.brownian(2, 200, 3, seed=s), dtype=torch.float64, device="cuda") for s in (741, 742))
    w = torch.ones(2, 2, dtype=torch.float64, device="cuda")
    kw = dict(scheme=scheme, degree=4, compute="f64")
    assert sk.device_status() == 0
    _, tape = sk.sigkernel_forward_tape(X, Y, **kw)
    want = sk.sigkernel_backward_tape(tape, w, X, Y, **kw)
    assert sk.device_status() == 0
    sk.set_wait_limit(1)
    try:
        sk.sigkernel_backward_tape(tape, w, X, Y, **kw)
        assert sk.device_status() == SK_ERR_DEVICE_TIMEOUT
    finally:
        sk.set_wait_limit(0)
    got = sk.sigkernel_backward_tape(tape, w, X, Y, **kw)
    assert sk.device_status() == 0
    for g, h in zip(got, want):
        assert (g - h).abs().max() <= 1e-12 * h.abs().max()  # FP64 sums in another order
