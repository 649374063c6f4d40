"""GPU parity of the finite-difference sweeps where a warp step covers a tile of R x C sub-cells:
steep paths, whose sub-cells have |m| from below to far above the bound up to which a tile is swept
without rescaling between its columns, at every tile shape (dyadic orders 0..5), for ragged lengths
of one and two strips and a single increment.

All increments are positive, so every node is positive and the schemes' updates only add: a value is
off by at most the number of updates on the way to it times 2^-24 in FP32 (fewer than 1600 nodes a
side at three operations each: 3e-4; rounding that is not all one way stays far below), and 2^-53
in FP64 (6e-13).  Tolerances: 1e-4 and 1e-11 relative, as the other FD comparisons use.
"""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu
sk = pytest.importorskip("paper_2502_08470_gb300.sigkernel")


@pytest.fixture(scope="module", autouse=True)
def _cuda_available():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _steep(L, d, mean_m, seed):
    """[L, d] points whose increments u satisfy <u, u'> about mean_m, all coordinates positive."""
    rng = np.random.default_rng(seed)
    inc = rng.uniform(0.5, 1.5, size=(L - 1, d)) * np.sqrt(mean_m / d)
    return np.concatenate([np.zeros((1, d)), np.cumsum(inc, 0)])


@pytest.mark.parametrize("scheme", ["fd1", "fd2"])
@pytest.mark.parametrize("lam", [0, 1, 2, 3, 4, 5])
@pytest.mark.parametrize("lx,ly", [(2, 2), (6, 37), (35, 5)])
def test_steep_paths(scheme, lam, lx, ly):
    for per_subcell in (0.3, 6.0):  # below and above the tile bound of |m| = 1
        x = _steep(lx, 3, per_subcell * 4 ** lam, 900 + lam)
        y = _steep(ly, 3, per_subcell * 4 ** lam, 950 + lam)
        ref = oracle.gram([x], [y], scheme, 2, lam)[0, 0]
        if not np.isfinite(ref):
            continue
        for compute, tol in (("f64", 1e-11), ("f32", 1e-4)):
            X, Y = (torch.tensor(v[None], device="cuda") for v in (x, y))
            k = sk.sigkernel_pairs(X, Y, [0], [0], scheme=scheme, dyadic=lam, compute=compute).item()
            assert sk.device_status() == 0
            assert abs(k - ref) <= tol * abs(ref)
            if lam <= 4 and lx * ly * 4 ** lam < 20000:
                g = np.array([1.0 / ref])
                gX, gY = sk.sigkernel_backward(torch.tensor(g, device="cuda"), X, Y, pair_a=[0], pair_b=[0],
                                               scheme=scheme, dyadic=lam, compute=compute)
                assert sk.device_status() == 0
                rx, ry = oracle.grad(x, y, scheme, 2, lam)
                for got, want in ((gX, rx), (gY, ry)):
                    want = want / ref
                    err = np.max(np.abs(got.cpu().numpy().reshape(want.shape) - want)) / np.max(np.abs(want))
                    assert err < (1e-9 if compute == "f64" else 1e-4)
