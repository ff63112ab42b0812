"""The measured cases: whole solves Z = r(tA) B through the package's public entry points.

Each case is one problem as a user of this framework poses it: an operator (a 1-D, 2-D or 3-D
convection-diffusion stencil, a symmetric Toeplitz matrix, a general sparse matrix), a block of
right-hand sides drawn from N(0, 1), a time, a precision, and the plan that is made once and kept.
The operators, sizes and options are those of ``paper_1405_0707_gb300.inputs`` and of the tests;
``draw`` spreads them over the ranges in between.  ``exact`` forms e^{tA} B in 64 bits: by the
closed-form eigenpairs of each axis for the stencils, by a Taylor series for the others (the
degree-14 rational approximation itself is within 2e-14 |B| of it).
"""
import math
import random

import numpy as np
import torch

from paper_1405_0707_gb300 import inputs
from paper_1405_0707_gb300.api import Batch, Plan, colmajor
from paper_1405_0707_gb300.autograd import expm_block


def _grid(name, sides, p, t, precision, diff, vel, m=10, tol=1e-10, own_stream=False, kind="grid"):
    s, v = list(sides) + [1, 1], list(vel) + [0.0, 0.0]
    return dict(name=name, kind=kind, ndim=len(sides), nx=s[0], ny=s[1], nz=s[2], vx=v[0], vy=v[1], vz=v[2],
                diff=diff, p=p, t=t, m=m, tol=tol, precision=precision, own_stream=own_stream)


def listed():
    return [
        # the smallest calls: one line of 2000 points, four columns (the 1-D heat equation);
        # nothing but launches and host round trips
        _grid("line-2000", (2000,), 4, 0.1, "fp64", 1.0, (0.0,)),
        # the paper's Example 5.1a: 2-D Poisson on 99^2, three columns, m = 30, tol 1e-8
        _grid("poisson-99", (99, 99), 3, 1.0, "fp64", 0.25, (0.0, 0.0), m=30, tol=1e-8),
        # the 256^2 convection-diffusion problem at its longest time: Algorithm 2, whose
        # (tA)^{-1} is the sine transforms and line solves
        _grid("grid2d-256-long", (256, 256), 8, 0.1, "mixed", 0.1, (1.0, 1.0)),
        # the same at its shortest time: Algorithm 1 (products with tA); a stepper that keeps
        # its solves on a stream of its own
        _grid("grid2d-256-short", (256, 256), 8, 1e-3, "mixed", 0.1, (1.0, 1.0), own_stream=True),
        # the default precision on that grid at its middle time
        _grid("grid2d-256-fp64", (256, 256), 8, 1e-2, "fp64", 0.1, (1.0, 1.0), own_stream=True),
        # an odd 3-D box with a few columns: ragged rows, ragged transforms
        _grid("grid3d-odd", (45, 72, 69), 3, 7.5e-3, "mixed", 1.0, (3.0, -5.0, 1.0)),
        # the largest 3-D instance: 96^3, 16 columns, 1.2 GB of basis
        _grid("grid3d-96", (96, 96, 96), 16, 0.01, "mixed", 1.0, (1.0, -1.0, 0.5), own_stream=True),
        # the large Toeplitz problem: n = 2^20, FFT products of length 2^21
        dict(name="toeplitz-1m", kind="toeplitz", n=1 << 20, bw=256, p=16, t=1.0, m=10, tol=1e-13, precision="mixed",
             own_stream=True),
        # a Toeplitz matrix of no particular size in the default precision
        dict(name="toeplitz-odd-fp64", kind="toeplitz", n=50021, bw=100, p=5, t=1.0, m=10, tol=1e-13, precision="fp64",
             own_stream=False),
        # a general sparse matrix with a 3-D grid's pattern and random values
        dict(name="csr-3d", kind="csr", nx=56, ny=48, nz=44, p=8, t=0.2, m=10, tol=1e-10, precision="mixed",
             own_stream=False),
        # a training step through torch autograd: L = |r(tA) B - Y|^2, 512 points along x as in the
        # differentiation workload, 32 columns, gradients for B and t
        _grid("grad-512x352", (512, 352), 32, 1e-2, "mixed", 0.1, (1.0, 1.0), kind="grad"),
        # many independent 3-D problems of all sizes, widths and times in one graph launch
        dict(name="batch-3d", kind="batch", count=12, shapes=7, m=10, tol=1e-10, precision="mixed", own_stream=True),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["line", "grid2d", "grid2d", "grid2d", "grid3d", "grid3d", "toeplitz", "csr", "grad", "batch"])
    precision = rng.choice(["mixed", "mixed", "fp64"])
    own = rng.random() < 0.5
    if kind == "line":
        return _unnamed(_grid("", (int(_log(rng, 200, 4000)),), rng.randint(1, 16), _log(rng, 0.03, 0.3), precision, 1.0,
                              (0.0,), own_stream=own))
    if kind == "grid2d":
        sides = (int(_log(rng, 40, 320)), int(_log(rng, 40, 320)))
        return _unnamed(_grid("", sides, rng.randint(1, 16), _log(rng, 1e-3, 0.2), precision, 0.1,
                              (rng.uniform(-1, 1), rng.uniform(-1, 1)), m=rng.choice([10, 10, 20]), own_stream=own))
    if kind == "grid3d":
        top = 96 if precision == "mixed" else 64
        sides = tuple(rng.randint(24, top) for _ in range(3))
        return _unnamed(_grid("", sides, rng.randint(1, 16), _log(rng, 1e-3, 0.05), precision, 1.0,
                              tuple(rng.uniform(-6, 6) for _ in range(3)), own_stream=own))
    if kind == "toeplitz":
        top = 1 << 20 if precision == "mixed" else 1 << 18
        return dict(kind="toeplitz", n=int(_log(rng, 4000, top)), bw=int(_log(rng, 8, 256)), p=rng.randint(1, 16),
                    t=_log(rng, 0.3, 3.0), m=10, tol=1e-13, precision=precision, own_stream=own)
    if kind == "csr":
        return dict(kind="csr", nx=rng.randint(20, 64), ny=rng.randint(20, 64), nz=rng.randint(20, 64),
                    p=rng.randint(1, 16), t=_log(rng, 0.05, 0.5), m=10, tol=1e-10, precision=precision, own_stream=own)
    if kind == "grad":
        return _unnamed(_grid("", (rng.randint(64, 384), rng.randint(64, 384)), rng.randint(4, 32),
                              _log(rng, 6e-3, 0.05), "mixed", 0.1, (rng.uniform(-1, 1), rng.uniform(-1, 1)), kind="grad"))
    return dict(kind="batch", count=rng.randint(4, 14), shapes=rng.randint(0, 1 << 30), m=10, tol=1e-10,
                precision="mixed", own_stream=True)


def _unnamed(case):
    return {k: v for k, v in case.items() if k != "name"}


def _sides(case):
    return tuple(case[k] for k in ("nx", "ny", "nz"))[:case.get("ndim", 3)]


def _vel(case):
    return tuple(case[k] for k in ("vx", "vy", "vz"))[:case.get("ndim", 3)]


def _instances(case):
    """The batch's problems as grid cases: sides 32..96, p 1..16, t from 1e-3 to 0.1, v ~ 5 N(0, I)
    with every cell Peclet number below 1 (the ranges of the batched workload, without the times
    at which the result has decayed below the approximation's own error)."""
    r = random.Random(case["shapes"])
    out = []
    while len(out) < case["count"]:
        sides = tuple(r.randint(32, 96) for _ in range(3))
        vel = tuple(5.0 * r.gauss(0.0, 1.0) for _ in range(3))
        p, t = r.randint(1, 16), 10.0 ** r.uniform(-3.0, -1.0)
        if all(abs(v) < 2.0 * (N + 1) and abs(v) < 12.0 for v, N in zip(vel, sides)):
            out.append(_grid("", sides, p, t, case["precision"], 1.0, vel, m=case["m"], tol=case["tol"]))
    return out


def _rhs(n, p, seed):
    """B: i.i.d. N(0, 1), n x p column-major on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((p, n), dtype=torch.float64, device="cuda", generator=g).T


def _target(case, seed):
    """Y of the training step: smooth columns, random combinations of the 4 x 4 lowest modes."""
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    c = torch.randn((case["p"], 4, 4), dtype=torch.float64, device="cuda", generator=g) * 0.02
    k = torch.arange(1, 5, dtype=torch.float64, device="cuda")
    sx, sy = (torch.sin(math.pi * torch.outer(k, torch.arange(1, N + 1, dtype=torch.float64, device="cuda") / (N + 1)))
              for N in (case["nx"], case["ny"]))
    return torch.einsum("pij,iy,jx->pyx", c, sy, sx).reshape(case["p"], -1).T


def _csr(case, seed):
    return inputs.sparse_stencil_matrix((case["nx"], case["ny"], case["nz"]), seed=seed)


def _size(case):
    return case["n"] if case["kind"] == "toeplitz" else math.prod(_sides(case))


def prepare(case, seed):
    kw = dict(m=case["m"], tol=case["tol"], max_cycles=400, precision=case["precision"])
    kind = case["kind"]
    if kind == "batch":
        probs = _instances(case)
        streams = [torch.cuda.Stream() for _ in probs]
        plans = [Plan(_sides(c), c["diff"], _vel(c), p_max=c["p"], stream=s, **kw) for c, s in zip(probs, streams)]
        Bs = [_rhs(math.prod(_sides(c)), c["p"], seed * 1000 + k) for k, c in enumerate(probs)]
        torch.cuda.synchronize()
        stream = torch.cuda.Stream()
        return dict(kind=kind, batch=Batch(plans, [c["t"] for c in probs], Bs, stream=stream),
                    keep=(plans, streams, stream))
    n, p = _size(case), case["p"]
    kw["stream"] = torch.cuda.Stream() if case["own_stream"] else None
    if kind == "toeplitz":
        plan = Plan.toeplitz(inputs.toeplitz_column(case["bw"]), n, p_max=p, **kw)
    elif kind == "csr":
        indptr, indices, data = _csr(case, seed)
        plan = Plan.csr((data, indices, indptr), p_max=p, **kw)
    else:
        plan = Plan(_sides(case), case["diff"], _vel(case), p_max=p, **kw)
    state = dict(kind=kind, plan=plan, t=case["t"], B=_rhs(n, p, seed), keep=kw["stream"])
    if kind == "grad":
        state["t"] = torch.tensor(case["t"], dtype=torch.float64, requires_grad=True)
        state["B"].requires_grad_()
        state["Y"] = _target(case, seed)
    else:
        state["Z"] = colmajor(n, p)
    torch.cuda.synchronize()
    return state


def run(state):
    if state["kind"] == "batch":
        return state["batch"].run()[0]
    if state["kind"] == "grad":
        Z = expm_block(state["t"], state["B"], state["plan"])
        loss = (Z - state["Y"]).square().sum()
        dt, dB = torch.autograd.grad(loss, (state["t"], state["B"]))
        return {"Z": Z.detach(), "loss": loss.detach(), "dB": dB, "dt": dt}
    return state["plan"].expm_block(state["t"], state["B"], state["Z"])[0]


def work(case):
    """B read and Z written once (with gradients also Y read and dL/dB written), and one product
    of the operator with the block, which no method does without."""
    if case["kind"] == "batch":
        each = [work(c) for c in _instances(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    np_ = _size(case) * case["p"]
    if case["kind"] == "toeplitz":
        N = 1 << (2 * case["n"] - 1).bit_length()
        return {"bytes": 16.0 * np_, "flops": 5.0 * N * math.log2(N) * case["p"]}
    points = {1: 3, 2: 5, 3: 7}[case.get("ndim", 3)]
    passes = 2.0 if case["kind"] == "grad" else 1.0
    extra = 12.0 * _size(case) * points if case["kind"] == "csr" else 0.0
    return {"bytes": 16.0 * np_ * passes + extra, "flops": 2.0 * points * np_ * passes}


# ---------------------------------------------------------------- the values in 64 bits
def _axis(N, diff, v):
    """(l, c, u) of one axis: tridiag(l, c, u) = diff Laplacian_h - v grad_h, zero boundary values."""
    h = 1.0 / (N + 1)
    return diff / h ** 2 + v / (2 * h), -2.0 * diff / h ** 2, diff / h ** 2 - v / (2 * h)


def _axis_exp(N, diff, v, t):
    """e^{t tridiag(l, c, u)} as a dense matrix from the closed-form eigenpairs, the eigenvalues
    without cancellation."""
    l, c, u = _axis(N, diff, v)
    s = math.sqrt(l * u)
    j = torch.arange(1, N + 1, dtype=torch.float64, device="cuda")
    lam = (v * (N + 1)) ** 2 / (c - 2 * s) - 4 * s * torch.sin(j * (math.pi / (2 * (N + 1)))) ** 2
    S = math.sqrt(2.0 / (N + 1)) * torch.sin(torch.outer(j, j).remainder(2 * (N + 1)) * (math.pi / (N + 1)))
    d = torch.exp((j - (N + 1) / 2) * (0.5 * math.log(l / u)))
    return (d[:, None] * S) @ (torch.exp(t * lam)[:, None] * S / d[None, :])


def _axis_matrix(N, diff, v):
    l, c, u = _axis(N, diff, v)
    one = torch.ones(N, dtype=torch.float64, device="cuda")
    return torch.diag(c * one) + torch.diag(l * one[1:], -1) + torch.diag(u * one[1:], 1)


def _along(X, mats, sides, total):
    """X (n x p) with mats[d] applied along axis d (x fastest): one after another, or summed."""
    T = X.T.reshape((X.shape[1],) + tuple(reversed(sides)))
    out = 0
    for d, M in enumerate(mats):
        Y = torch.movedim(torch.movedim(T, -1 - d, -1) @ M.T, -1, -1 - d)
        if total:
            out = out + Y
        else:
            T = Y
    return (out if total else T).reshape(X.shape[1], -1).T


def _grid_exact(case, X, sign=1.0):
    sides, vel = _sides(case), _vel(case)
    return _along(X, [_axis_exp(N, case["diff"], sign * v, case["t"]) for N, v in zip(sides, vel)], sides, False)


def _taylor(apply, X, t, radius):
    """e^{tM} X by steps of |t| radius <= 1, radius a bound of |M + radius I|: the series of M + radius I."""
    steps = max(1, math.ceil(t * radius))
    h = t / steps
    for _ in range(steps):
        term, total = X, X.clone()
        for k in range(1, 26):
            term = (apply(term) + radius * term) * (h / k)
            total += term
        X = total * math.exp(-h * radius)
    return X


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return [_grid_exact(c, _rhs(math.prod(_sides(c)), c["p"], seed * 1000 + k)) for k, c in enumerate(_instances(case))]
    n, p = _size(case), case["p"]
    B = _rhs(n, p, seed)
    if kind == "toeplitz":
        a = torch.from_numpy(np.asarray(inputs.toeplitz_column(case["bw"]))).cuda()
        col = torch.zeros(2 * n, dtype=torch.float64, device="cuda")
        col[:len(a)] = a
        col[2 * n - len(a) + 1:] = a[1:].flip(0)
        lam = torch.fft.rfft(col).real
        apply = lambda X: torch.fft.irfft(torch.fft.rfft(X.T, n=2 * n) * lam, n=2 * n)[:, :n].T  # noqa: E731
        return _taylor(apply, B, case["t"], 1.6)
    if kind == "csr":
        indptr, indices, data = _csr(case, seed)
        M = torch.sparse_csr_tensor(torch.from_numpy(indptr), torch.from_numpy(indices.astype(np.int64)),
                                    torch.from_numpy(data), size=(n, n), dtype=torch.float64, device="cuda")
        diag = -float(np.min(data))     # the largest |a_ii|: every Gershgorin disc lies in |z + diag| <= diag
        return _taylor(lambda X: M @ X, B.contiguous(), case["t"], diag)
    Z = _grid_exact(case, B)
    if kind == "grid":
        return Z
    D = Z - _target(case, seed)
    AZ = _along(Z, [_axis_matrix(N, case["diff"], v) for N, v in zip(_sides(case), _vel(case))], _sides(case), True)
    return {"Z": Z, "loss": D.square().sum(), "dB": _grid_exact(case, 2.0 * D, -1.0), "dt": 2.0 * (D * AZ).sum()}
