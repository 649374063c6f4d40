"""FP64 FD calls on short paths, a refined column at a time (fd_narrow), against the tile of several columns: a
short pair alone, and the same pair in a set whose longest path makes the call take tiles.  Both form the
same sub-cells in the same order: values, also those of the forward that records a tape, are equal
bit for bit.  Gradients differ by the order of the sums over a cell's sub-cells (and, in the set, by
zeros added): to 1e-12 of their scale, in FP64.
"""
import pytest
import torch

from paper_2502_08470_gb300 import workloads as W

pytestmark = pytest.mark.gpu
sk = pytest.importorskip("paper_2502_08470_gb300.sigkernel")


@pytest.fixture(scope="module", autouse=True)
def _cuda_available():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _sets(px, py, d=3):
    x, y = W.brownian(1, px, d, seed=600)[0], W.brownian(1, py, d, seed=601)[0]
    long = W.brownian(1, 200, d, seed=602)[0]
    return [[sk.Paths.from_list([p]) for p in (x, y)], [sk.Paths.from_list([p, long]) for p in (x, y)]]


@pytest.mark.parametrize("scheme", ["fd1", "fd2", "fd_implicit"])
@pytest.mark.parametrize("lam", [0, 1, 2, 3, 4, 5])
@pytest.mark.parametrize("px,py", [(2, 2), (9, 30), (33, 33), (34, 20)])
def test_narrow_equals_tiles(scheme, lam, px, py):
    few, many = _sets(px, py)
    kw = dict(scheme=scheme, degree=0, dyadic=lam, compute="f64")
    a = sk.sigkernel_pairs(*few, [0], [0], **kw)
    b = sk.sigkernel_pairs(*many, [0, 1], [0, 1], strip_pipeline=False, **kw)
    assert sk.device_status() == 0
    assert torch.equal(a, b[:1])


@pytest.mark.parametrize("scheme", ["fd1", "fd2", "fd_implicit"])
@pytest.mark.parametrize("lam", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("px,py", [(2, 3), (33, 33), (34, 20)])
def test_narrow_gradients(scheme, lam, px, py):
    few, many = _sets(px, py)
    kw = dict(scheme=scheme, degree=0, dyadic=lam, compute="f64")
    w = torch.tensor([1.7, 0.0], dtype=torch.float64, device="cuda")
    k0, tape = sk.sigkernel_forward_tape(*few, pair_a=[0], pair_b=[0], **kw)
    g0 = sk.sigkernel_backward_tape(tape, w[:1], *few, pair_a=[0], pair_b=[0], **kw)
    k1, tape = sk.sigkernel_forward_tape(*many, pair_a=[0, 1], pair_b=[0, 1], **kw)
    g1 = sk.sigkernel_backward_tape(tape, w, *many, pair_a=[0, 1], pair_b=[0, 1], **kw)
    assert sk.device_status() == 0
    assert torch.equal(k0, k1[:1])
    for a, b, n in zip(g0, g1, (px, py)):
        assert (a - b[:n]).abs().max() <= 1e-12 * a.abs().max()
