"""FP64 pairs of one strip with their cells split over four warps (sk_fwd_split.cuh) against one warp
per pair: the same sums in the same order, so equal bit for bit, at every order the split serves, from
one cell to a full strip, with refinement and wide increments, over ragged sets with empty pairs."""
import pytest
import torch

from paper_2502_08470_gb300 import workloads as W

pytestmark = pytest.mark.gpu
sk = pytest.importorskip("paper_2502_08470_gb300.sigkernel")


@pytest.fixture(scope="module", autouse=True)
def _cuda_available():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("scheme", ["approx", "interp"])
@pytest.mark.parametrize("N", [2, 3, 4, 5, 6, 7, 8, 9])
@pytest.mark.parametrize("lx,ly,d,lam", [(2, 2, 1, 0), (33, 33, 2, 0), (20, 90, 5, 0), (9, 5, 17, 2)])
def test_split_equals_one_warp(scheme, N, lx, ly, d, lam):
    xs = [p[:max(1, lx - i)] for i, p in enumerate(W.brownian(4, lx, d, seed=1))]
    ys = [p[:max(1, ly - 3 * i)] for i, p in enumerate(W.brownian(3, ly, d, seed=2))]
    X, Y = sk.Paths.from_list(xs), sk.Paths.from_list(ys)
    kw = dict(scheme=scheme, degree=N, dyadic=lam, compute="f64")
    got = sk.sigkernel_gram(X, Y, **kw)
    want = sk.sigkernel_gram(X, Y, strip_pipeline=False, **kw)
    assert sk.device_status() == 0
    assert torch.equal(got, want)
