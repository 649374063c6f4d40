"""GPU tests of the strip chain (a warp per strip, sk_chain.cuh) against one warp per pair.

Both run the same cells in the same order, with M formed in the same order, so values are equal bit
for bit; gradients differ only by the order of the contraction's atomics (FP64 sums, and in FP32
its shared column sums too).  Shapes at the edges: rows that
fill or just exceed a strip, fewer columns than a batch or a tile of M, wide and narrow increments,
refinement, orders whose hand-off column takes 2 to 17 units, ragged sets, and hand-off buffers too
few to hold every pair at once (a smaller workspace: pairs in groups, buffers used in turn).
"""
import numpy as np
import pytest
import torch

from paper_2502_08470_gb300 import workloads as W

pytestmark = pytest.mark.gpu
sk = pytest.importorskip("paper_2502_08470_gb300.sigkernel")


@pytest.fixture(scope="module", autouse=True)
def _cuda_available():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _cuda(a):
    return torch.as_tensor(np.asarray(a), dtype=torch.float64, device="cuda")


def _both(X, Y, pa, pb, **kw):
    out = [sk.sigkernel_pairs(X, Y, pa, pb, strip_pipeline=f, tensor_cores=False, tiled_m=False, **kw) for f in (True, False)]
    assert sk.device_status() == 0
    return out


@pytest.mark.parametrize("scheme,N", [("approx", 2), ("approx", 5), ("approx", 16), ("interp", 4), ("interp", 12)])
@pytest.mark.parametrize("compute", ["f32", "f64"])
@pytest.mark.parametrize("lx,ly,d,lam", [(33, 2, 1, 0), (34, 9, 3, 0), (65, 17, 8, 0), (66, 130, 17, 0), (66, 20, 32, 0), (97, 64, 33, 0),
                                         (21, 19, 4, 2)])
def test_chain_equals_one_warp(scheme, N, compute, lx, ly, d, lam):
    X = _cuda(W.brownian(3, lx, d, seed=1))
    Y = _cuda(W.brownian(2, ly, d, seed=2))
    a, b = _both(X, Y, [0, 1, 2, 2], [1, 0, 1, 0], scheme=scheme, degree=N, dyadic=lam, compute=compute)
    assert torch.equal(a, b)


@pytest.mark.parametrize("compute", ["f32", "f64"])
def test_large_exponents(compute):
    """Kernels far beyond FP32's range: the chain hands exponents on and aligns them."""
    u = np.linspace(0, 1, 97)[:, None] * np.full((1, 3), 18.0)
    a, b = _both(_cuda(u[None]), _cuda(u[None] * 1.1), [0], [0], degree=8, compute=compute)
    assert torch.equal(a, b) and a.item() > 1e20


def test_ragged_and_small_workspace():
    """Lengths from one point to several strips; then the same with a workspace whose hand-off buffers
    hold a few pairs at a time."""
    xs = [p[:n] for p, n in zip(W.brownian(60, 700, 4, seed=3), np.random.default_rng(4).integers(1, 700, 60))]
    ys = [p[:n] for p, n in zip(W.brownian(60, 600, 4, seed=5), np.random.default_rng(6).integers(1, 600, 60))]
    X, Y = sk.Paths.from_list(xs), sk.Paths.from_list(ys)
    a, b = _both(X, Y, list(range(60)), list(range(60)), compute="f32")
    assert torch.equal(a, b)
    G = sk.sigkernel_gram(X, Y, compute="f32", strip_pipeline=True, tensor_cores=False)
    full = sk.gram_workspace(X, Y, compute="f32", strip_pipeline=True).numel()
    sizes = 0
    for k in range(12):  # down to what one warp per pair needs, and no further
        ws = torch.empty(full >> k, dtype=torch.uint8, device="cuda")
        try:
            H = sk.sigkernel_gram(X, Y, compute="f32", strip_pipeline=True, tensor_cores=False, workspace=ws)
        except sk.SigKernelError as e:
            assert e.code == -4  # SK_ERR_WORKSPACE
            break
        assert sk.device_status() == 0
        assert torch.equal(G, H)
        sizes += 1
    assert sizes >= 4


@pytest.mark.parametrize("scheme,N", [("approx", 3), ("approx", 6), ("interp", 5)])
@pytest.mark.parametrize("lx,ly,d,lam", [(34, 3, 2, 0), (98, 41, 5, 0), (40, 70, 20, 1)])
def test_chained_gradients(scheme, N, lx, ly, d, lam):
    """Three pairs (chained, in the tape forward and in the adjoint).  FP64 gradients against the same
    three within a batch large enough for one warp per pair (the others have a zero upstream
    gradient); FP32 tape-forward values against one warp per pair, bit for bit, and FP32 gradients
    against the FP64 ones to 1e-4 of their scale, as the FP32 adjoints are held to everywhere."""
    X = _cuda(W.brownian(3, lx, d, seed=7))
    Y = _cuda(W.brownian(3, ly, d, seed=8))
    kw = dict(scheme=scheme, degree=N, dyadic=lam, tensor_cores=False)
    w = torch.tensor([0.7, -1.3, 2.0], dtype=torch.float64, device="cuda")
    few = sk.sigkernel_backward(w, X, Y, pair_a=[0, 1, 2], pair_b=[1, 2, 0], compute="f64", **kw)
    n = 3000
    pa = torch.arange(n) % 3
    wn = torch.zeros(n, dtype=torch.float64, device="cuda")
    wn[:3] = w
    many = sk.sigkernel_backward(wn, X, Y, pair_a=pa, pair_b=(pa + 1) % 3, compute="f64", **kw)
    for g, h in zip(few, many):
        assert (g - h).abs().max() <= 1e-12 * h.abs().max()
    K, tape = sk.sigkernel_forward_tape(X, Y, pair_a=[0, 1, 2], pair_b=[1, 2, 0], compute="f32", **kw)
    assert torch.equal(K, _both(X, Y, [0, 1, 2], [1, 2, 0], scheme=scheme, degree=N, dyadic=lam, compute="f32")[1])
    g32 = sk.sigkernel_backward_tape(tape, w, X, Y, pair_a=[0, 1, 2], pair_b=[1, 2, 0], compute="f32", **kw)
    assert sk.device_status() == 0
    for g, h in zip(g32, few):
        assert (g - h).abs().max() <= 1e-4 * h.abs().max()
