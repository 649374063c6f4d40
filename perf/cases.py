"""Performance cases of the signature-kernel library: the calls a user's program makes, over the range
of sizes it makes them at.

A case names a job (``pairs``, ``gram``, ``train``, ``mmd``), a scheme with its order and dyadic
refinement, the compute type, and the shape and law of the paths.  ``prepare`` draws the paths on
the GPU, ``run`` is one pass through the public entry points (``sigkernel_pairs``,
``sigkernel_gram``, ``SigKernel.gram`` and ``SigKernel.mmd2`` with their gradients), and ``exact``
is the same scheme evaluated cell by cell in 64-bit torch.

The library returns values in float64 whatever the compute type.  A program that asks for FP32
compute works in its inputs' type, so the values of those cases are handed on as float32.
"""
from __future__ import annotations

import math
from fractions import Fraction

import torch

from paper_2502_08470_gb300 import sigkernel as sk

DTYPES = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}


def listed():
    base = dict(scheme="approx", degree=6, dyadic=0, compute="f32", dtype="f32", law="brownian", symmetric=False)
    return [
        # One pair of short 2-d paths with the plain method in FP64: an interactive call, all latency.
        dict(base, name="pair_f64", job="pairs", nx=1, ny=1, length=33, d=2, degree=4, compute="f64", dtype="f64"),
        # Kernel matrix of a data set of short multivariate series, as a kernel classifier needs it.
        dict(base, name="symmetric_f32", job="gram", nx=150, ny=150, length=100, d=3, symmetric=True),
        # The plain FP64 Gram: the library's default compute type, where accuracy comes first.
        dict(base, name="gram_f64", job="gram", nx=64, ny=64, length=129, d=8, compute="f64", dtype="f64"),
        # The headline step: a 128 x 128 Gram and its gradients inside a training loop.
        dict(base, name="gram_train_f32", job="train", nx=128, ny=128, length=257, d=8),
        # A batch of highly oscillatory pairs with the interpolation scheme.
        dict(base, name="osc_f32", job="pairs", nx=64, ny=64, length=1025, d=4, scheme="interp", degree=8, law="osc"),
        # Training on a small batch of long oscillatory paths: few pairs, each a long chain.
        dict(base, name="osc_train_f32", job="train", nx=8, ny=8, length=513, d=4, scheme="interp", degree=8,
             law="osc"),
        # A ragged batch: lengths log-uniform over a factor of 64, BF16 points.
        dict(base, name="uneven_bf16", job="pairs", nx=4096, ny=4096, length=4096, shortest=64, d=16, dtype="bf16",
             law="uneven"),
        # One step of a generative model trained on (unbiased) MMD^2 with a mini-batch of short paths.
        dict(base, name="mmd_batch_f32", job="mmd", nx=16, ny=16, length=65, d=5),
        # MMD^2 and its gradients between two large samples of wide paths.
        dict(base, name="mmd_train_f32", job="mmd", nx=128, ny=128, length=257, d=32),
        # The second-order finite-difference scheme, refined twice: the baseline most programs use.
        dict(base, name="fd_gram_f32", job="gram", nx=128, ny=128, length=129, d=8, scheme="fd2", degree=0, dyadic=2),
        # The same scheme differentiated, refined once.
        dict(base, name="fd_train_f32", job="train", nx=48, ny=48, length=129, d=8, scheme="fd2", degree=0, dyadic=1),
        # One pair of very long paths (a tick-by-tick series against another).
        dict(base, name="long_f32", job="pairs", nx=1, ny=1, length=16385, d=4),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _cost(case):
    """Multiply-adds of a case, FP64 ones at their rate on this GPU (about 1/64 of FP32's, rounded up)."""
    return _flops(case) * (76 if case["compute"] == "f64" else 1)


def draw(rng):
    """One case of the listed ones' ranges: a kind of call, then sizes spread over its range."""
    while True:
        c = _draw_any(rng)
        if _cost(c) <= 1.2e12:
            return c


def _draw_any(rng):
    base = dict(scheme="approx", degree=6, dyadic=0, compute="f32", dtype="f32", law="brownian", symmetric=False)
    kind = rng.choice(["pair_f64", "gram_f64", "gram", "train", "osc", "osc_train", "uneven", "mmd", "fd", "fd_train",
                       "long"])
    if kind == "pair_f64":
        n = _log_int(rng, 1, 64)
        scheme = rng.choice(["approx", "interp"])
        return dict(base, job="pairs", nx=n, ny=n, length=_log_int(rng, 10, 200), d=rng.randint(1, 4), scheme=scheme,
                    degree=rng.choice([4, 6, 8]), compute="f64", dtype="f64")
    if kind == "gram_f64":
        return dict(base, job="gram", nx=_log_int(rng, 8, 64), ny=_log_int(rng, 8, 64), length=_log_int(rng, 20, 257),
                    d=rng.randint(2, 10), degree=rng.choice([4, 5, 6, 8]), compute="f64", dtype="f64")
    if kind == "gram":
        n, sym = _log_int(rng, 8, 200), rng.random() < 0.5
        return dict(base, job="gram", nx=n, ny=n if sym else _log_int(rng, 8, 200), length=_log_int(rng, 20, 400),
                    d=_log_int(rng, 1, 32), degree=rng.choice([4, 5, 6, 7, 8]), symmetric=sym)
    if kind == "train":
        return dict(base, job="train", nx=_log_int(rng, 8, 128), ny=_log_int(rng, 8, 128), length=_log_int(rng, 20, 257),
                    d=_log_int(rng, 2, 32), degree=rng.choice([4, 5, 6, 8]))
    if kind == "osc":
        n = _log_int(rng, 8, 64)
        return dict(base, job="pairs", nx=n, ny=n, length=_log_int(rng, 129, 1025), d=rng.randint(2, 4),
                    scheme="interp", degree=rng.choice([6, 7, 8]), law="osc")
    if kind == "osc_train":
        return dict(base, job="train", nx=_log_int(rng, 2, 8), ny=_log_int(rng, 2, 8), length=_log_int(rng, 65, 513),
                    d=rng.randint(2, 4), scheme="interp", degree=rng.choice([6, 7, 8]), law="osc")
    if kind == "uneven":
        n = _log_int(rng, 256, 4096)
        return dict(base, job="pairs", nx=n, ny=n, length=_log_int(rng, 512, 4096), shortest=_log_int(rng, 16, 64),
                    d=_log_int(rng, 3, 32), dtype=rng.choice(["bf16", "f32"]), law="uneven")
    if kind == "mmd":
        return dict(base, job="mmd", nx=_log_int(rng, 8, 128), ny=_log_int(rng, 8, 128), length=_log_int(rng, 33, 257),
                    d=_log_int(rng, 2, 32), degree=rng.choice([4, 5, 6]))
    if kind == "fd":
        return dict(base, job="gram", nx=_log_int(rng, 8, 128), ny=_log_int(rng, 8, 128), length=_log_int(rng, 20, 257),
                    d=_log_int(rng, 2, 16), scheme=rng.choice(["fd1", "fd2"]), degree=0, dyadic=rng.randint(0, 3))
    if kind == "fd_train":
        return dict(base, job="train", nx=_log_int(rng, 8, 64), ny=_log_int(rng, 8, 64), length=_log_int(rng, 20, 200),
                    d=_log_int(rng, 2, 16), scheme=rng.choice(["fd1", "fd2"]), degree=0, dyadic=rng.randint(0, 2))
    n = rng.randint(1, 2)
    return dict(base, job="pairs", nx=n, ny=n, length=_log_int(rng, 4097, 16385 if n == 1 else 8193),
                d=rng.randint(2, 8), degree=rng.choice([4, 6]))


# ----------------------------------------------------------------------------------------------
# Inputs
# ----------------------------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _generator(seed, salt):
    return torch.Generator(device=_device()).manual_seed(int(seed) * 7 + salt)


def _dense(case, n, g, drift=0.0, vol=1.0):
    """[n, L, d] points in the case's type: Brownian motion on [0, 1], or noisy sines with
    frequencies U(10, 200) and phases U(0, 2 pi)."""
    L, d, dev = case["length"], case["d"], _device()
    if case["law"] == "osc":
        t = torch.linspace(0.0, 1.0, L, dtype=torch.float64, device=dev).view(1, L, 1)
        w = 10.0 + 190.0 * torch.rand(n, 1, d, dtype=torch.float64, device=dev, generator=g)
        phi = 2.0 * math.pi * torch.rand(n, 1, d, dtype=torch.float64, device=dev, generator=g)
        eps = torch.randn(n, L, d, dtype=torch.float64, device=dev, generator=g) * math.sqrt(1e-3)
        # a quarter of unit amplitude: programs scale such paths so that the kernel stays in the
        # range of their type (unit amplitudes reach 1e42)
        x = 0.25 * (torch.sin(w * t + phi) + eps)
    else:
        x = torch.randn(n, L, d, dtype=torch.float64, device=dev, generator=g) * (vol / math.sqrt(L - 1)) + drift / (L - 1)
        x[:, 0] = 0.0
        x = x.cumsum(1)
    return x.to(DTYPES[case["dtype"]])


def _ragged(case, n, g):
    """n Brownian paths as rows and offsets, lengths log-uniform in [shortest, length], increments
    N(0, 1/length)."""
    dev, d = _device(), case["d"]
    lo, hi = math.log(case["shortest"]), math.log(case["length"])
    lens = torch.exp(lo + (hi - lo) * torch.rand(n, dtype=torch.float64, device=dev, generator=g)).floor().long()
    lens.clamp_(case["shortest"], case["length"])
    off = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    off[1:] = lens.cumsum(0)
    owner = torch.repeat_interleave(torch.arange(n, device=dev), lens)
    x = torch.randn(owner.numel(), d, dtype=torch.float64, device=dev, generator=g) / lens[owner].sqrt().unsqueeze(1)
    x[off[:-1]] = 0.0
    x = x.cumsum(0)
    x = x - x[off[:-1]][owner]
    return x.to(DTYPES[case["dtype"]]), off


def _inputs(case, seed):
    gx, gy = _generator(seed, 1), _generator(seed, 2)
    if case["law"] == "uneven":
        return _ragged(case, case["nx"], gx), _ragged(case, case["ny"], gy)
    X = _dense(case, case["nx"], gx)
    if case["symmetric"]:
        return X, X
    # an MMD compares a sample with one of another law
    Y = _dense(case, case["ny"], gy, 0.5, 1.2) if case["job"] == "mmd" else _dense(case, case["ny"], gy)
    return X, Y


def _upstream(case, seed):
    """Upstream gradient of a Gram (what the rest of a loss hands back)."""
    return torch.randn(case["nx"], case["ny"], dtype=torch.float64, device=_device(), generator=_generator(seed, 3))


def prepare(case, seed):
    X, Y = _inputs(case, seed)
    opts = dict(scheme=case["scheme"], degree=case["degree"], dyadic=case["dyadic"], compute=case["compute"])
    s = {"job": case["job"], "opts": opts, "hold": torch.float32 if case["compute"] == "f32" else torch.float64}
    if case["law"] == "uneven":
        X = sk.Paths(X[0], X[1], case["length"])
        Y = sk.Paths(Y[0], Y[1], case["length"])
    if case["job"] == "pairs":
        s["pair"] = torch.arange(case["nx"], dtype=torch.int64, device=_device())
    elif case["job"] in ("train", "mmd"):
        X, Y = X.requires_grad_(), Y.requires_grad_()
        s["kernel"] = sk.SigKernel(**opts)
        if case["job"] == "train":
            s["up"] = _upstream(case, seed)
    s["X"], s["Y"] = X, None if case["symmetric"] else Y
    return s


def run(s):
    X, Y, hold = s["X"], s["Y"], s["hold"]
    if s["job"] == "pairs":
        return sk.sigkernel_pairs(X, Y, s["pair"], s["pair"], **s["opts"]).to(hold)
    if s["job"] == "gram":
        return sk.sigkernel_gram(X, Y, **s["opts"]).to(hold)
    if s["job"] == "train":
        K = s["kernel"].gram(X, Y)
        gX, gY = torch.autograd.grad(K, (X, Y), s["up"])
        return {"K": K.detach().to(hold), "gX": gX, "gY": gY}
    m = s["kernel"].mmd2(X, Y, unbiased=True)
    gX, gY = torch.autograd.grad(m, (X, Y))
    return {"mmd2": m.detach().to(hold), "gX": gX, "gY": gY}


# ----------------------------------------------------------------------------------------------
# What a pass cannot do without
# ----------------------------------------------------------------------------------------------
def _cells(case):
    """(pairs, cells before refinement) of a case."""
    if case["law"] == "uneven":
        lo, hi = case["shortest"], case["length"]
        mean = (hi - lo) / math.log(hi / lo) - 1 if hi > lo else hi - 1  # of a log-uniform length
        return case["nx"], case["nx"] * mean * mean
    inc = case["length"] - 1
    nx, ny = case["nx"], case["ny"]
    if case["job"] == "pairs":
        pairs = nx
    elif case["job"] == "mmd":
        pairs = nx * (nx + 1) // 2 + ny * (ny + 1) // 2 + nx * ny
    else:
        pairs = nx * (nx + 1) // 2 if case["symmetric"] else nx * ny
    return pairs, pairs * inc * inc


def _flops(case):
    _, cells = _cells(case)
    sub = 4 ** case["dyadic"]
    N = case["degree"]
    if case["scheme"] in ("fd1", "fd2"):
        cell = 6 * sub
    elif case["scheme"] == "approx":  # both edges: couplings N (N + 1), convolution N (N - 1) / 2, scaling N
        cell = 2 * 2 * (N * (N + 1) + N * (N - 1) // 2 + N) * sub
    else:  # the same series with 6 more terms, and their projection onto N + 1 coefficients
        cell = 2 * 2 * (N * (N + 7) + N * (N - 1) // 2 + 6 * N + N + 6 + 6 * (N + 1)) * sub
    dot = 2 * case["d"]
    if case["job"] in ("train", "mmd"):  # the adjoint of the cell, and the two contractions of dk/dM
        return cells * (2 * cell + 3 * dot)
    return cells * (cell + dot)


def work(case):
    size = {"f64": 8, "f32": 4, "bf16": 2}[case["dtype"]]
    pairs, _ = _cells(case)
    if case["law"] == "uneven":
        lo, hi = case["shortest"], case["length"]
        rows = 2 * case["nx"] * ((hi - lo) / math.log(hi / lo) if hi > lo else hi)
    else:
        rows = (case["nx"] + (0 if case["symmetric"] else case["ny"])) * case["length"]
    data = rows * case["d"] * size
    values = {"pairs": case["nx"], "mmd": 1}.get(case["job"], case["nx"] * case["ny"]) * (8 if case["compute"] == "f64" else 4)
    moved = data + values
    if case["job"] in ("train", "mmd"):
        moved += data  # the gradients
    if case["job"] == "train":
        moved += case["nx"] * case["ny"] * 8  # the upstream gradient
    return {"bytes": moved, "flops": _flops(case)}


# ----------------------------------------------------------------------------------------------
# The schemes in 64 bits, one antidiagonal of every pair at a time
# ----------------------------------------------------------------------------------------------
def _projection(N, J):
    """[N + 1, J]: the factorial-scaled coefficients of the interpolant, at the N + 1 Chebyshev
    extrema of [0, 1], of u^j / j! for j = N + 1 .. N + J (exact rationals: at those points the
    shifted Chebyshev polynomial of degree N + r equals the one of degree N - r)."""
    cheb = [[Fraction(1)], [Fraction(-1), Fraction(2)]]  # T*_k(u) = T_k(2u - 1)
    for k in range(2, N + 1):
        a, b = cheb[-1], cheb[-2]
        new = [Fraction(0)] * (k + 1)
        for i, v in enumerate(a):
            new[i] -= 2 * v
            new[i + 1] += 4 * v
        for i, v in enumerate(b):
            new[i] -= v
        cheb.append(new)
    P = torch.zeros(N + 1, J, dtype=torch.float64)
    for j in range(N + 1, N + J + 1):
        mono = [Fraction(0)] * (N + 1)
        for k in range(j + 1):  # u^j = sum_k c_k T*_k
            c = Fraction(math.comb(2 * j, j - k) * (1 if k == 0 else 2), 4 ** j)
            m = k % (2 * N)
            for i, v in enumerate(cheb[m if m <= N else 2 * N - m]):
                mono[i] += c * v
        for i in range(N + 1):
            P[i, j - N - 1] = float(mono[i] * math.factorial(i) / math.factorial(j))
    return P


class _Poly:
    """Cell map of the polynomial schemes on factorial-scaled edge coefficients (bottom a, left b):
    c_n = sum_{k<=n} (.)_k e_{n-k} + e_n sum_{k>=1} (other)_k n!/(n+k)!, e_m = M^m / m!."""

    def __init__(self, scheme, N, dev):
        self.N, self.interp = N, scheme == "interp"
        self.NE = N + 14 if self.interp else N
        H = torch.zeros(self.NE + 1, N + 1, dtype=torch.float64)
        for n in range(self.NE + 1):
            for k in range(1, N + 1):
                H[n, k] = math.factorial(n) / math.factorial(n + k)
        self.H = H.to(dev)
        self.P = _projection(N, self.NE - N).to(dev) if self.interp else None
        self.end = torch.tensor([0.5 / math.factorial(n) for n in range(self.NE + 1)], dtype=torch.float64, device=dev)
        self.inv = torch.tensor([1.0] + [1.0 / m for m in range(1, self.NE + 1)], dtype=torch.float64, device=dev)

    def start(self, P, R, dev):
        S = torch.zeros(2, self.N + 1, P, R + 1, dtype=torch.float64, device=dev)
        S[:, 0] = 1.0
        return S

    def _series(self, M):
        e = M.unsqueeze(0) * self.inv.view(-1, 1, 1)
        e[0] = 1.0
        return e.cumprod(0)

    def _couple(self, S):
        h = torch.einsum("nk,ekpl->enpl", self.H, S.flip(0))
        return h

    def series(self, S, M):
        """All terms c [2, NE + 1, P, l] of the outgoing (top, right) edges."""
        e, N = self._series(M), self.N
        c = self._couple(S) * e
        for m in range(self.NE + 1):  # the convolution, one shift at a time
            top = min(N, self.NE - m)
            c[:, m:m + top + 1].addcmul_(S[:, :top + 1], e[m].expand_as(S[:, :top + 1]))
        if self.interp:  # the right edge's corner term is the bottom edge's constant
            c[1] += (S[0, 0] - S[1, 0]) * e
        return c

    def project(self, c):
        if not self.interp:
            return c
        return c[:, :self.N + 1] + torch.einsum("nj,ejpl->enpl", self.P, c[:, self.N + 1:])

    def project_t(self, cb):
        if not self.interp:
            return cb
        return torch.cat([cb, torch.einsum("nj,enpl->ejpl", self.P, cb)], 1)

    def adjoint(self, S, M, cb):
        """Adjoints of the incoming edges and of M from those of all outgoing terms."""
        e, N = self._series(M), self.N
        eb = (self._couple(S) * cb).sum(0)
        Sb = torch.einsum("nk,enpl->ekpl", self.H, cb * e).flip(0).contiguous()
        for m in range(self.NE + 1):
            top = min(N, self.NE - m)
            part = cb[:, m:m + top + 1]
            Sb[:, :top + 1].addcmul_(part, e[m].expand_as(part))
            eb[m] += (part * S[:, :top + 1]).sum((0, 1))
        if self.interp:
            d = S[0, 0] - S[1, 0]
            eb += cb[1] * d
            g = (cb[1] * e).sum(0)
            Sb[0, 0] += g
            Sb[1, 0] -= g
        return Sb, (eb[1:] * e[:-1]).sum(0)


def _poly(case, dX, dY, lx, ly, weight):
    """Values and, with `weight` (one per pair), gradients with respect to the refined increments
    [P, R, d] and [P, C, d] of pairs with lx x ly cells."""
    dev = dX.device
    P, R, C = dX.shape[0], dX.shape[1], dY.shape[1]
    cell = _Poly(case["scheme"], case["degree"], dev)
    S = cell.start(P, R, dev)
    flip = dY.flip(1)
    out = torch.ones(P, dtype=torch.float64, device=dev)
    ends = {}
    for p, t in enumerate((lx + ly - 2).tolist()):
        ends.setdefault(t, []).append(p)
    saved = []

    def slices(t):
        lo, hi = max(0, t - C + 1), min(t, R - 1)
        x = dX[:, lo:hi + 1]
        y = flip[:, C - 1 - t + lo:C - t + hi]  # column t - i beside row i
        return lo, hi, x, y

    for t in range(R + C - 1):
        lo, hi, x, y = slices(t)
        M = (x * y).sum(-1)
        cur = S[..., lo:hi + 1]
        if weight is not None:
            cur = cur.clone()
            saved.append((cur, M))
        c = cell.series(cur, M)
        if t in ends:
            idx = torch.tensor(ends[t], device=dev)
            at = c[:, :, idx, lx[idx] - 1 - lo]
            out[idx] = (at * cell.end.view(1, -1, 1)).sum((0, 1))
        c = cell.project(c)
        S[0, :, :, lo:hi + 1] = c[0]
        S[1, :, :, lo + 1:hi + 2] = c[1]
    if weight is None:
        return out, None, None
    gX, gY = torch.zeros_like(dX), torch.zeros_like(dY)
    Sb = torch.zeros_like(S)
    gflip = gY.flip(1)
    for t in range(R + C - 2, -1, -1):
        lo, hi, x, y = slices(t)
        cb = cell.project_t(torch.stack([Sb[0, :, :, lo:hi + 1], Sb[1, :, :, lo + 1:hi + 2]]))
        if t in ends:
            idx = torch.tensor(ends[t], device=dev)
            cb[:, :, idx, lx[idx] - 1 - lo] += cell.end.view(1, -1, 1) * weight[idx].view(1, 1, -1)
        cur, M = saved.pop()
        sb, mb = cell.adjoint(cur, M, cb)
        Sb[1, :, :, lo + 1:hi + 2] = 0.0
        Sb[..., lo:hi + 1] = sb
        gX[:, lo:hi + 1] += mb.unsqueeze(-1) * y
        gflip[:, C - 1 - t + lo:C - t + hi] += mb.unsqueeze(-1) * x
    return out, gX, gflip.flip(1)


def _fd(case, dX, dY, weight):
    """The explicit finite-difference schemes: with s = k10 + k01,
    k11 = s - k00 + (m / 2) s + w (s + k00), w = 0 (first order) or m^2 / 12 (second order)."""
    dev = dX.device
    P, R, C = dX.shape[0], dX.shape[1], dY.shape[1]
    second = case["scheme"] == "fd2"
    flip = dY.flip(1)
    old = torch.ones(P, R + 1, dtype=torch.float64, device=dev)  # nodes (i, t - i)
    new = torch.ones(P, R + 1, dtype=torch.float64, device=dev)  # nodes (i, t + 1 - i)
    saved = []

    def slices(t):
        lo, hi = max(0, t - C + 1), min(t, R - 1)
        return lo, hi, dX[:, lo:hi + 1], flip[:, C - 1 - t + lo:C - t + hi]

    for t in range(R + C - 1):
        lo, hi, x, y = slices(t)
        m = (x * y).sum(-1)
        k00, s = old[:, lo:hi + 1].clone(), new[:, lo + 1:hi + 2] + new[:, lo:hi + 1]
        w = m * m / 12 if second else torch.zeros_like(m)
        k11 = s - k00 + 0.5 * m * s + w * (s + k00)
        if weight is not None:
            saved.append((m, k00, s))
        old, new = new, torch.ones_like(new)
        new[:, lo + 1:hi + 2] = k11
        if hi < R - 1:
            new[:, hi + 2:] = 1.0
    value = new[:, R].clone()
    if weight is None:
        return value, None, None
    gX, gflip = torch.zeros_like(dX), torch.zeros_like(flip)
    nb = torch.zeros(P, R + 1, dtype=torch.float64, device=dev)  # adjoints of the nodes of step t
    nb[:, R] = weight
    ob = torch.zeros_like(nb)
    pb = torch.zeros_like(nb)
    for t in range(R + C - 2, -1, -1):
        lo, hi, x, y = slices(t)
        m, k00, s = saved.pop()
        g = nb[:, lo + 1:hi + 2]
        w = m * m / 12 if second else torch.zeros_like(m)
        dw = m / 6 if second else torch.zeros_like(m)
        mb = g * (0.5 * s + dw * (s + k00))
        sb = g * (1 + 0.5 * m + w)
        ob[:, lo + 1:hi + 2] += sb
        ob[:, lo:hi + 1] += sb
        pb[:, lo:hi + 1] += g * (w - 1)
        gX[:, lo:hi + 1] += mb.unsqueeze(-1) * y
        gflip[:, C - 1 - t + lo:C - t + hi] += mb.unsqueeze(-1) * x
        nb, ob, pb = ob, pb, torch.zeros_like(pb)
    return value, gX, gflip.flip(1)


def _solve(case, dX, dY, lx, ly, weight):
    r = 1 << case["dyadic"]
    if r > 1:
        dX = dX.repeat_interleave(r, 1) / r
        dY = dY.repeat_interleave(r, 1) / r
    if case["scheme"] in ("fd1", "fd2"):
        v, gX, gY = _fd(case, dX, dY, weight)
    else:
        v, gX, gY = _poly(case, dX, dY, lx * r, ly * r, weight)
    if gX is not None and r > 1:
        gX = gX.view(gX.shape[0], -1, r, gX.shape[2]).sum(2) / r
        gY = gY.view(gY.shape[0], -1, r, gY.shape[2]).sum(2) / r
    return v, gX, gY


def _points_grad(g):
    """Gradients with respect to points from those with respect to increments, [n, L - 1, d]."""
    z = torch.zeros_like(g[:, :1])
    return torch.cat([z, g], 1) - torch.cat([g, z], 1)


def _block(case, X, Y, weight):
    """K [nx, ny] and, with `weight` [nx, ny], the gradients of sum(weight * K) by the points."""
    dX, dY = X.double().diff(dim=1), Y.double().diff(dim=1)
    nx, ny = X.shape[0], Y.shape[0]
    a = torch.arange(nx, device=X.device).repeat_interleave(ny)
    b = torch.arange(ny, device=X.device).repeat(nx)
    r = 1 << case["dyadic"]
    cells = dX.shape[1] * dY.shape[1] * r * r
    words = (3 if case["scheme"] in ("fd1", "fd2") else 2 * case["degree"] + 3) * cells if weight is not None else \
        64 * (dX.shape[1] + dY.shape[1]) * r
    step = int(max(1, min(a.numel(), 4e9 // words)))
    K = torch.empty(nx, ny, dtype=torch.float64, device=X.device)
    gX, gY = torch.zeros_like(dX), torch.zeros_like(dY)
    for k in range(0, a.numel(), step):
        i, j = a[k:k + step], b[k:k + step]
        lx = torch.full((i.numel(),), dX.shape[1], device=X.device)
        ly = torch.full((i.numel(),), dY.shape[1], device=X.device)
        v, gx, gy = _solve(case, dX[i], dY[j], lx, ly, None if weight is None else weight[i, j])
        K[i, j] = v
        if weight is not None:
            gX.index_add_(0, i, gx)
            gY.index_add_(0, j, gy)
    return K, _points_grad(gX), _points_grad(gY)


def _padded(rows, off, paths, longest):
    """[P, longest, d] increments of the given paths of a ragged set, zero past their end."""
    d = rows.double().diff(dim=0)
    at = off[paths].unsqueeze(1) + torch.arange(longest, device=rows.device)
    keep = at < (off[paths + 1] - 1).unsqueeze(1)
    return d[at.clamp(max=d.shape[0] - 1)] * keep.unsqueeze(-1)


def exact(case, seed):
    """What ``run`` returns, from the schemes' definitions in 64-bit torch."""
    X, Y = _inputs(case, seed)
    if case["law"] == "uneven":
        (rx, ox), (ry, oy) = X, Y
        lx, ly = ox.diff() - 1, oy.diff() - 1
        order = torch.argsort(lx + ly, descending=True)
        out = torch.empty(case["nx"], dtype=torch.float64, device=rx.device)
        k = 0
        while k < order.numel():  # the longest pairs first, more of them at once as they get shorter
            longest = int(max(lx[order[k:]].max(), ly[order[k:]].max()))
            n = int(max(32, min(order.numel() - k, 4e8 // (longest * (2 * case["degree"] + 2 + 2 * case["d"])))))
            p = order[k:k + n]
            R, C = int(lx[p].max()), int(ly[p].max())
            out[p] = _solve(case, _padded(rx, ox, p, R), _padded(ry, oy, p, C), lx[p], ly[p], None)[0]
            k += n
        return out
    if case["job"] == "pairs":
        dX, dY = X.double().diff(dim=1), Y.double().diff(dim=1)
        n = torch.full((X.shape[0],), X.shape[1] - 1, device=X.device)
        return _solve(case, dX, dY, n, n, None)[0]
    if case["job"] == "gram":
        return _block(case, X, Y, None)[0]
    if case["job"] == "train":
        K, gX, gY = _block(case, X, Y, _upstream(case, seed))
        return {"K": K, "gX": gX, "gY": gY}
    # the unbiased estimate: the diagonals of the two samples' own Grams stay out
    nx, ny = case["nx"], case["ny"]
    ones = lambda a, b: torch.ones(a, b, dtype=torch.float64, device=X.device)  # noqa: E731
    Wxx = (ones(nx, nx) - torch.eye(nx, dtype=torch.float64, device=X.device)) / (nx * (nx - 1))
    Wyy = (ones(ny, ny) - torch.eye(ny, dtype=torch.float64, device=X.device)) / (ny * (ny - 1))
    Wxy = ones(nx, ny) * (-2.0 / (nx * ny))
    Kxx, a0, a1 = _block(case, X, X, Wxx)
    Kyy, b0, b1 = _block(case, Y, Y, Wyy)
    Kxy, c0, c1 = _block(case, X, Y, Wxy)
    return {"mmd2": (Kxx * Wxx).sum() + (Kyy * Wyy).sum() + (Kxy * Wxy).sum(), "gX": a0 + a1 + c0, "gY": b0 + b1 + c1}
