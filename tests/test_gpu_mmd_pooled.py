"""MMD^2 of sets swept as one pooled Gram (their longest paths about equally long) against the three
blocks computed on their own: sigkernel_gram for the values, sigkernel_backward for the gradients.

The sets are ragged, do not start at their buffer's first row or end at its last, and have lengths on
either side of the bound for pooling.  The values are FP64 sums of the same Gram entries, off by at most
the number of terms times 2^-53 of their magnitude (1e-12); gradients sum the same dk/dM in another
order: 1e-12 of their scale in FP64, and in FP32, whose row and column sums are FP32, 1e-5.
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


def _set(lens, d, seed, lead, tail):
    """Ragged Paths whose rows have `lead` unused rows before the first path and `tail` after the last."""
    x = W.brownian(len(lens), max(lens), d, seed=seed)
    rows = np.concatenate([np.full((lead, d), 7.0)] + [x[i, :n] for i, n in enumerate(lens)] + [np.full((tail, d), -3.0)])
    off = lead + np.concatenate([[0], np.cumsum(lens)])
    return sk.Paths(torch.tensor(rows, device="cuda"), torch.tensor(off, dtype=torch.int64, device="cuda"), max(lens))


@pytest.mark.parametrize("compute,vtol,gtol", [("f64", 1e-12, 1e-12), ("f32", 1e-12, 1e-5)])
@pytest.mark.parametrize("unbiased", [False, True])
@pytest.mark.parametrize("la,lb", [([20, 1, 33, 7], [30, 41, 2]), ([40, 12], [50, 3, 50]), ([40, 12], [51, 3, 50])])
@pytest.mark.parametrize("scheme,N,d", [("approx", 4, 3), ("approx", 6, 9), ("fd2", 0, 2), ("interp", 4, 2)])
def test_pooled_sets(compute, vtol, gtol, unbiased, la, lb, scheme, N, d):
    A, B = _set(la, d, 1, 3, 2), _set(lb, d, 2, 0, 5)
    kw = dict(scheme=scheme, degree=N, compute=compute, dyadic=1 if scheme == "fd2" else 0)
    m, parts, gA, gB = sk.sigkernel_mmd2(A, B, unbiased=unbiased, grads=True, **kw)
    m0, parts0 = sk.sigkernel_mmd2(A, B, unbiased=unbiased, **kw)
    Kaa, Kbb, Kab = (sk.sigkernel_gram(*p, **kw) for p in ((A, None), (B, None), (A, B)))
    assert sk.device_status() == 0
    na, nb = len(la), len(lb)
    waa = torch.full((na, na), 1.0 / (na * (na - unbiased)), dtype=torch.float64, device="cuda")
    wbb = torch.full((nb, nb), 1.0 / (nb * (nb - unbiased)), dtype=torch.float64, device="cuda")
    wab = torch.full((na, nb), -2.0 / (na * nb), dtype=torch.float64, device="cuda")
    if unbiased:
        waa.fill_diagonal_(0.0)
        wbb.fill_diagonal_(0.0)
    means = torch.stack([(Kaa * waa).sum(), (Kbb * wbb).sum(), -0.5 * (Kab * wab).sum()])
    scale = means.abs().max().item()
    tol = vtol if compute == "f64" else 2e-5  # (FP32: M from the tensor cores or not, by the batch's size)
    for p in (parts, parts0):
        assert (p - means).abs().max().item() <= tol * scale
    assert abs(m.item() - m0.item()) <= tol * scale
    ra, _ = sk.sigkernel_backward(waa, A, None, **kw)
    rb, _ = sk.sigkernel_backward(wbb, B, None, **kw)
    ca, cb = sk.sigkernel_backward(wab, A, B, **kw)
    assert sk.device_status() == 0
    for got, want in ((gA, ra + ca), (gB, rb + cb)):
        assert (got - want).abs().max() <= gtol * want.abs().max()
