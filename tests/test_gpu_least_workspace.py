"""Every call in the least workspace that it takes (sigkernel_workspace_least), where the planned one holds
the buffers of a strip chain: the same values; and calls that find no room for the planned one, in
the binding (the allocation fails) and in the library (no workspace given, from a memory pool too small).
"""
import ctypes

import pytest
import torch

from paper_2502_08470_gb300 import workloads as W

pytestmark = pytest.mark.gpu
sk = pytest.importorskip("paper_2502_08470_gb300.sigkernel")


@pytest.fixture(scope="module", autouse=True)
def _cuda_available():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _paths(n, points, d, seed):
    return torch.as_tensor(W.brownian(n, points, d, seed=seed), dtype=torch.float32, device="cuda")


def _small(empty, seen):
    """torch.empty that has no room for a planned workspace: the first of two sizes asked for fails."""
    def alloc(*size, **kw):
        if kw.get("dtype") == torch.uint8 and len(size) == 1 and not seen.get("failed"):
            seen["failed"] = size[0]
            raise torch.cuda.OutOfMemoryError("no room")
        t = empty(*size, **kw)
        if kw.get("dtype") == torch.uint8 and seen.get("failed") and "got" not in seen:
            seen["got"] = t.numel()
        return t
    return alloc


@pytest.mark.parametrize("scheme,d", [("approx", 3), ("approx", 8), ("interp", 3)])
def test_calls_without_room_for_a_chain(monkeypatch, scheme, d):
    X, Y = _paths(6, 700, d, 751), _paths(5, 650, d, 752)
    kw = dict(scheme=scheme, degree=4, compute="f32")
    w = torch.ones(6, 5, dtype=torch.float64, device="cuda")
    labels = sk.split_labels(7, 6, 5)
    _, tape = sk.sigkernel_forward_tape(X, Y, **kw)
    calls = {
        "pairs": lambda: sk.sigkernel_pairs(X, Y, [0, 1, 2], [2, 1, 0], **kw),
        "gram": lambda: sk.sigkernel_gram(X, Y, **kw),
        "tape": lambda: sk.sigkernel_forward_tape(X, Y, tape=tape, **kw)[0],
        "backward_tape": lambda: sk.sigkernel_backward_tape(tape, w, X, Y, **kw),
        "backward": lambda: sk.sigkernel_backward(w, X, Y, **kw),
        "mmd2": lambda: sk.sigkernel_mmd2(X, Y, grads=True, **kw),
        "mmd2 value": lambda: sk.sigkernel_mmd2(X, Y, **kw),
        "mmd2_test": lambda: sk.sigkernel_mmd2_test(X, Y, labels=labels, **kw),
    }
    for name, call in calls.items():
        want = call()
        seen = {}
        with monkeypatch.context() as m:
            m.setattr(torch, "empty", _small(torch.empty, seen))
            got = call()
        assert sk.device_status() == 0
        assert seen["got"] < seen["failed"], name
        for g, h in zip(*((v,) if isinstance(v, torch.Tensor) else v for v in (got, want))):
            assert (g - h).abs().max() <= (1e-4 if "backward" in name or name == "mmd2" else 1e-6) * h.abs().max(), name


class _PoolProps(ctypes.Structure):  # CUmemPoolProps
    _fields_ = [("alloc_type", ctypes.c_int), ("handle_types", ctypes.c_int), ("location_type", ctypes.c_int),
                ("location_id", ctypes.c_int), ("security", ctypes.c_void_p), ("max_size", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


def test_library_without_room_for_a_chain():
    """sigkernel_gram without a workspace, from a pool of 64 MiB, where its plan with a chain takes more: it runs
    with the least one."""
    X, Y = sk.as_paths(_paths(8, 1025, 4, 753)), sk.as_paths(_paths(8, 1025, 4, 754))
    cX, cY = sk._cpaths(X), sk._cpaths(Y)
    opt = sk._options("approx", 6, 0, "f32", 0)
    lib, cu, ref = sk.load_library(), ctypes.CDLL("libcuda.so.1"), ctypes.byref
    want = sk.sigkernel_gram(X, Y, degree=6, compute="f32")
    size, least = ctypes.c_size_t(0), ctypes.c_size_t(0)
    sk._check(lib.sigkernel_workspace_size(sk.OP_GRAM, ref(cX), ref(cY), 4, ctypes.c_int64(-1), ref(opt), ref(size)))
    sk._check(lib.sigkernel_workspace_least(sk.OP_GRAM, ref(cX), ref(cY), 4, ctypes.c_int64(-1), ref(opt), ref(least)))
    assert least.value < 32 << 20 and size.value > 96 << 20
    got = torch.zeros_like(want)
    torch.cuda.synchronize()
    dev = torch.cuda.current_device()
    props = _PoolProps(alloc_type=1, location_type=1, location_id=dev, max_size=64 << 20)  # pinned, on the device
    pool, default = ctypes.c_void_p(), ctypes.c_void_p()
    assert cu.cuMemPoolCreate(ref(pool), ref(props)) == 0
    assert cu.cuDeviceGetDefaultMemPool(ref(default), dev) == 0
    assert cu.cuDeviceSetMemPool(dev, pool) == 0
    try:
        rc = lib.sigkernel_gram(ref(cX), ref(cY), 4, 1, ref(opt), got.data_ptr(), None, 0,
                                torch.cuda.current_stream().cuda_stream)
        message = lib.sigkernel_last_error()
        torch.cuda.synchronize()
    finally:
        cu.cuDeviceSetMemPool(dev, default)
        cu.cuMemPoolDestroy(pool)
    assert rc == 0, message
    assert sk.device_status() == 0
    assert torch.equal(got, want)
