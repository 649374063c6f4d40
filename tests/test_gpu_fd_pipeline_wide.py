"""The pipelined FD forward at lambda = 0 in FP32 with increments of one, two, three and more 16-byte chunks (more
than two go by another form of the inner product) against one warp per pair: the same products in the
same order, equal bit for bit."""
import pytest
import torch

from paper_2502_08470_gb300 import workloads as W

pytestmark = pytest.mark.gpu
sk = pytest.importorskip("paper_2502_08470_gb300.sigkernel")


@pytest.mark.parametrize("scheme", ["fd1", "fd2", "fd_implicit"])
@pytest.mark.parametrize("compute", ["f32", "f64"])
@pytest.mark.parametrize("d", [1, 4, 5, 8, 9, 12, 13, 33])
def test_pipeline_equals_one_warp(scheme, compute, d):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    X, Y = (torch.as_tensor(W.brownian(n, p, d, seed=801 + p), dtype=torch.float64, device="cuda") for n, p in ((3, 140), (2, 70)))
    kw = dict(scheme=scheme, degree=0, compute=compute)
    a, b = (sk.sigkernel_gram(X, Y, strip_pipeline=f, **kw) for f in (True, False))
    assert sk.device_status() == 0
    assert torch.equal(a, b)
