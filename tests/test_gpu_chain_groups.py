"""GPU tests of the strip chain where its buffers do not hold everything at once: a pair whose strips use
fewer buffers than it has hand-offs in turn, and pairs in several groups that take the two halves of the
buffers in turn, with waits that last longer than the limit on polls; and two calls at once on two streams.

A workspace smaller than the plan's leaves fewer buffers; that the chain still runs in it (and not one
warp per pair) shows in a limit of one poll, which only a chain's waits can exhaust.  The same cells
in the same order: equal bit for bit.
"""
import pytest
import torch

from paper_2502_08470_gb300 import workloads as W

pytestmark = pytest.mark.gpu
sk = pytest.importorskip("paper_2502_08470_gb300.sigkernel")

SK_ERR_DEVICE_TIMEOUT = -5


@pytest.fixture(scope="module", autouse=True)
def _cuda_available():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _paths(n, points, d, seed):
    return torch.as_tensor(W.brownian(n, points, d, seed=seed), dtype=torch.float64, device="cuda")


def _units(N, compute):
    words = (N + 1) * (1 if compute == "f32" else 2) + (1 if compute == "f32" else 0)
    return (words + 1) // 2


def _chained(X, Y, ws, kw):
    sk.set_wait_limit(1)
    try:
        sk.sigkernel_gram(X, Y, strip_pipeline=True, workspace=ws, **kw)
        torch.cuda.synchronize()
    finally:
        sk.set_wait_limit(0)
    return sk.device_status() == SK_ERR_DEVICE_TIMEOUT


@pytest.mark.parametrize("compute,N,drop", [("f32", 6, 40), ("f32", 2, 63), ("f64", 4, 1)])
def test_buffers_used_in_turn(compute, N, drop):
    """128 strips, 127 hand-offs, `drop` buffers fewer."""
    X, Y = _paths(1, 4097, 2, 701), _paths(1, 301, 2, 702)
    kw = dict(degree=N, compute=compute, tensor_cores=False)
    full = sk.gram_workspace(X, Y, degree=N, compute=compute, strip_pipeline=True).numel()
    ws = torch.empty(full - drop * 304 * _units(N, compute) * 16, dtype=torch.uint8, device="cuda")
    assert sk.device_status() == 0
    got = sk.sigkernel_gram(X, Y, strip_pipeline=True, workspace=ws, **kw)
    assert sk.device_status() == 0
    assert torch.equal(got, sk.sigkernel_gram(X, Y, strip_pipeline=False, **kw))
    assert _chained(X, Y, ws, kw)


@pytest.mark.parametrize("scheme,N,compute,limit", [("interp", 12, "f64", 1 << 15), ("approx", 6, "f32", 0)])
def test_groups(scheme, N, compute, limit):
    """Nine pairs of 14 strips, one to each half of the buffers: nine groups.  With the slow FP64 steps a
    pair takes about 50 ms and the limit's polls about 20, so the wait of a group's first strip for the
    group before the last goes on only because strips finish meanwhile."""
    X, Y = _paths(3, 430, 2, 703), _paths(3, 301, 2, 704)
    kw = dict(scheme=scheme, degree=N, compute=compute, tensor_cores=False)
    full = sk.gram_workspace(X, Y, scheme=scheme, degree=N, compute=compute, strip_pipeline=True).numel()
    pair = 13 * 304 * _units(N, compute) * 16  # hand-off bytes of a pair
    ws = torch.empty(full - 9 * pair + 2 * pair + pair // 2, dtype=torch.uint8, device="cuda")
    assert sk.device_status() == 0
    sk.set_wait_limit(limit)
    try:
        got = sk.sigkernel_gram(X, Y, strip_pipeline=True, workspace=ws, **kw)
        torch.cuda.synchronize()
    finally:
        sk.set_wait_limit(0)
    assert sk.device_status() == 0
    assert torch.equal(got, sk.sigkernel_gram(X, Y, strip_pipeline=False, **kw))
    assert _chained(X, Y, ws, kw)


def test_two_streams():
    """Two chains at once, each with a workspace that the other does not see."""
    sets = [(_paths(2, 700 + 90 * k, 3, 710 + k), _paths(3, 400, 3, 720 + k)) for k in range(2)]
    want = [sk.sigkernel_gram(X, Y, compute="f32", strip_pipeline=False, tensor_cores=False) for X, Y in sets]
    ws = [sk.gram_workspace(X, Y, compute="f32", strip_pipeline=True) for X, Y in sets]
    got = [torch.zeros_like(w) for w in want]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    for _ in range(4):
        for (X, Y), w, g, s in zip(sets, ws, got, streams):
            with torch.cuda.stream(s):
                sk.sigkernel_gram(X, Y, compute="f32", strip_pipeline=True, tensor_cores=False, workspace=w, out=g)
    torch.cuda.synchronize()
    assert sk.device_status() == 0
    for g, w in zip(got, want):
        assert torch.equal(g, w)
