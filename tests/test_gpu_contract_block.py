"""GPU test of the FP32 contraction for up to 8 coordinates, where a lane takes a block of 8 x 4 cells
of a 32 x 32 tile: rows and columns at the edges of tiles and of the accumulator's window (1024
columns), few and all coordinates, refinement, the polynomial and the FD tapes.  FP32 gradients are held
to the FP64 ones, whose contraction walks rows and columns one by one: 1e-4 of their scale, the bar
of the FP32 adjoints everywhere.
"""
import numpy as np
import pytest
import torch

from paper_2502_08470_gb300 import workloads as W

pytestmark = pytest.mark.gpu
sk = pytest.importorskip("paper_2502_08470_gb300.sigkernel")


@pytest.mark.parametrize("rows,cols,lam", [(1, 1, 0), (3, 31, 0), (31, 33, 0), (32, 32, 0), (33, 64, 0), (64, 97, 0), (65, 5, 0),
                                           (40, 1030, 0), (17, 33, 1), (9, 50, 2)])
@pytest.mark.parametrize("d", [1, 4, 5, 8])
@pytest.mark.parametrize("scheme,N", [("approx", 5), ("fd2", 0)])
def test_block_contraction(rows, cols, lam, d, scheme, N):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    X = torch.as_tensor(W.brownian(2, rows + 1, d, seed=580 + d), device="cuda")
    Y = torch.as_tensor(W.brownian(3, cols + 1, d, seed=590 + d), device="cuda")
    w = torch.as_tensor(np.random.default_rng(581).uniform(0.5, 1.5, size=(2, 3)), device="cuda")
    kw = dict(scheme=scheme, degree=N, dyadic=lam)
    got, ref = (sk.sigkernel_backward(w, X, Y, compute=c, **kw) for c in ("f32", "f64"))
    assert sk.device_status() == 0
    for g, h in zip(got, ref):
        assert torch.isfinite(g).all()
        assert (g - h).abs().max() <= 1e-4 * h.abs().max()
