"""MMD^2 with gradients between sets of very different lengths (three blocks, whose contractions take different
amounts of shared memory): every compute type and order of the sets against the same sums from Grams and
their gradients, FP64 to 1e-10 and FP32 to 1e-4 of the scale, as gradients are held to everywhere."""
import pytest
import torch

from paper_2502_08470_gb300 import workloads as W

pytestmark = pytest.mark.gpu
sk = pytest.importorskip("paper_2502_08470_gb300.sigkernel")


@pytest.mark.parametrize("compute,tol", [("f64", 1e-10), ("f32", 1e-4)])
@pytest.mark.parametrize("scheme,N", [("approx", 6), ("interp", 4), ("fd2", 0)])
@pytest.mark.parametrize("pa,pb,d", [(9, 4, 8), (4, 9, 8), (300, 5, 3), (40, 200, 12)])
def test_gradients_of_unequal_sets(compute, tol, scheme, N, pa, pb, d):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    na, nb = 7, 5
    A = torch.as_tensor(W.brownian(na, pa, d, seed=791), dtype=torch.float64, device="cuda")
    B = torch.as_tensor(W.brownian(nb, pb, d, seed=792), dtype=torch.float64, device="cuda")
    kw = dict(scheme=scheme, degree=N)
    m, _, gA, gB = sk.sigkernel_mmd2(A, B, grads=True, compute=compute, tensor_cores=False, **kw)
    assert sk.device_status() == 0
    ones = lambda *shape: torch.ones(*shape, dtype=torch.float64, device="cuda")
    K = [sk.sigkernel_gram(X, Y, compute="f64", **kw) for X, Y in ((A, None), (B, None), (A, B))]
    want = K[0].mean() + K[1].mean() - 2 * K[2].mean()
    gaa = sk.sigkernel_backward(ones(na, na) / na**2, A, compute="f64", **kw)[0]
    gbb = sk.sigkernel_backward(ones(nb, nb) / nb**2, B, compute="f64", **kw)[0]
    gab = sk.sigkernel_backward(-2 * ones(na, nb) / (na * nb), A, B, compute="f64", **kw)
    scale = max(k.abs().max() for k in K)
    assert abs(m - want) <= tol * scale
    for got, parts in ((gA, (gaa, gab[0])), (gB, (gbb, gab[1]))):
        ref = sum(p.reshape(-1, d) for p in parts)
        assert (got - ref).abs().max() <= tol * max(p.abs().max() for p in parts)


@pytest.mark.parametrize("compute,tol", [("f64", 1e-11), ("f32", 1e-5)])
@pytest.mark.parametrize("na,nb", [(180, 20), (90, 90)])
def test_values_of_many_short_pairs(compute, tol, na, nb):
    """Sets on either side of the number of pairs from which on the value alone is taken from three blocks."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    A = torch.as_tensor(W.brownian(na, 12, 5, seed=793), dtype=torch.float64, device="cuda")
    B = torch.as_tensor(W.brownian(nb, 14, 5, seed=794), dtype=torch.float64, device="cuda")
    m, means = sk.sigkernel_mmd2(A, B, degree=6, compute=compute)
    K = [sk.sigkernel_gram(X, Y, degree=6, compute="f64").mean() for X, Y in ((A, None), (B, None), (A, B))]
    assert sk.device_status() == 0
    for got, want in zip(means, K):
        assert abs(got - want) <= tol * abs(want)
    assert abs(m - (K[0] + K[1] - 2 * K[2])) <= 4 * tol * max(K)
