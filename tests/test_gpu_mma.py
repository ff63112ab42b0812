"""The register-streamed tensor-core passes of the mixed path (k_mma.cu, rows_qr.cuh), through the
C ABI, against the CUDA-core row kernels and the oracle.

The sizes cover each N-tile width (p <= 8, <= 16, <= 32) and its edges, bases that end inside a
16-column chunk or pass the 240-column segment of the exact sums, row counts below one 16-row tile
and ragged against 16, 32 and 128 rows, and starting blocks that are localised (unit vectors, one
digit scale for every column) or spread out.

Tolerances, from the arithmetic: W - V h is exact to 2^-55 of each column's largest entry and the
forward substitution to ~2^-48 per product with the factor's condition below 300, so the relation
(tA)^{-1} V_m = V_{m+1} H~_m holds to 1e-12 relative; the projections carry 2^-25 per product, so
orthogonality and the agreement of H~ with the CUDA-core passes stay at FP32 level (1e-5, 1e-6, the
bounds of those passes' own tests).
"""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import cf, operators as ops, psbfom as ps
from paper_1405_0707_gb300 import inputs
from tests.gpu_util import need_gpu, rel, to_dev, to_np

pytestmark = pytest.mark.gpu


def _arnoldi(sides, p, m, V1, t):
    from paper_1405_0707_gb300 import Plan
    vel = (1.0, -0.5, 0.3)[:len(sides)]
    plan = Plan(sides, 0.1, vel, p_max=p, m=m, precision="mixed")
    Vg, Hg = plan.arnoldi(t, to_dev(V1))
    W = np.column_stack([to_np(plan.prec_apply(t, Vg[:, j * p:(j + 1) * p])) for j in range(m)])
    out = to_np(Vg), to_np(Hg), W
    plan.close()
    return out


@pytest.mark.parametrize("local", [False, True])
@pytest.mark.parametrize("sides,p,m", [((13,), 1, 3), ((47, 3), 3, 8), ((61, 59), 8, 10), ((33, 31, 29), 9, 5),
                                       ((97, 83), 16, 10), ((64, 40), 17, 6), ((130, 65), 32, 10), ((40, 41), 24, 3),
                                       ((70, 66), 16, 30), ((129, 127), 1, 40)])
def test_relation_orthogonality_and_h(sides, p, m, local, monkeypatch):
    need_gpu()
    n, t = int(np.prod(sides)), 0.05
    if local:
        V1 = np.zeros((n, p), order="F")
        V1[np.linspace(0, n - 1, p).astype(int), np.arange(p)] = 1.0
    else:
        V1, _ = ps.qr_positive(inputs.rhs(n, p, 8))
    V, H, W = _arnoldi(sides, p, m, V1, t)
    assert np.linalg.norm(W - V @ H) <= 1e-12 * np.linalg.norm(W)
    assert np.linalg.norm(V.T @ V - np.eye((m + 1) * p)) <= 1e-5
    monkeypatch.setenv("EXPM_CGS_TC", "0")
    Hr = _arnoldi(sides, p, m, V1, t)[1]
    k = p * min(m, 6)       # later columns amplify either side's FP32-level differences
    assert np.linalg.norm(H[:, :k] - Hr[:, :k]) <= 1e-6 * np.linalg.norm(Hr[:, :k])


@pytest.mark.parametrize("sides,p,t", [((256, 256), 8, 0.1), ((90, 77), 32, 0.03), ((40, 37, 35), 13, 0.02),
                                       ((300,), 5, 0.1)])
@pytest.mark.parametrize("repeated", [False, True])
def test_converged_solve_matches_closed_form(sides, p, t, repeated):
    """repeated: equal right-hand-side columns, which keep every block on the fallback passes."""
    need_gpu()
    from paper_1405_0707_gb300 import Plan
    n, d = int(np.prod(sides)), len(sides)
    diff, vel = (0.1, (1.0, 1.0)) if d == 2 else (1.0, (2.0, -1.0, 1.5)[:d])
    B = inputs.rhs(n, p, 44)
    if repeated:
        B[:, -1] = B[:, 0]
    Z, info = Plan(sides, diff, vel, p_max=p, m=10, tol=1e-11, max_cycles=400, precision="mixed").expm_block(t, to_dev(B))
    assert info.converged == 1
    ref = ops.exact_r_of_A_B(sides, diff, vel, t, cf.load_table(), B)
    assert rel(to_np(Z), ref) <= 1e-9, rel(to_np(Z), ref)


@pytest.mark.parametrize("local", [False, True])
@pytest.mark.parametrize("sides,p,m", [((401, 251), 1, 12), ((317, 106), 3, 6), ((130, 113), 8, 17), ((97, 83), 13, 10),
                                       ((83, 79), 16, 9), ((61, 59), 29, 6), ((33, 31, 29), 4, 5)])
def test_fp64_digit_passes_reach_fp64_rounding(sides, p, m, local):
    """FP64 plans with at least 100000 block entries: projections, updates and the Cholesky-QR products
    by digits.  Every product carries both operands to 2^-62 of their column's largest entry and is
    rounded once, so the relation holds to ~ (m p) eps of |W| and the basis is orthonormal to ~ (m p) p
    eps, the bounds of the FP64 kernels (1e-13 with the constants of these sizes).  The widths cover
    each N-tile size and bases that end inside a chunk or pass the 128-column segment."""
    need_gpu()
    from paper_1405_0707_gb300 import Plan
    n, t = int(np.prod(sides)), 0.05
    assert n * p >= 100000
    if local:
        V1 = np.zeros((n, p), order="F")
        V1[np.linspace(0, n - 1, p).astype(int), np.arange(p)] = 1.0
    else:
        V1, _ = ps.qr_positive(inputs.rhs(n, p, 8))
    plan = Plan(sides, 0.1, (1.0, -0.5, 0.3)[:len(sides)], p_max=p, m=m)
    Vg, Hg = plan.arnoldi(t, to_dev(V1))
    W = np.column_stack([to_np(plan.prec_apply(t, Vg[:, j * p:(j + 1) * p])) for j in range(m)])
    V, H = to_np(Vg), to_np(Hg)
    plan.close()
    assert np.linalg.norm(W - V @ H) <= 1e-13 * np.linalg.norm(W)
    assert np.linalg.norm(V.T @ V - np.eye((m + 1) * p)) <= 1e-13


def _times_longdouble(A, X):
    A, Y = A.tocsr(), np.zeros(X.shape, dtype=np.longdouble)
    X = X.astype(np.longdouble)
    for k in range(int(np.diff(A.indptr).max())):
        rows = np.nonzero(np.diff(A.indptr) > k)[0]
        idx = A.indptr[rows] + k
        Y[rows] += A.data[idx].astype(np.longdouble)[:, None] * X[A.indices[idx]]
    return Y


@pytest.mark.parametrize("local", [False, True])
@pytest.mark.parametrize("sides,diff,vel,t,p", [((256, 256), 0.1, (1.0, -0.5), 1e-2, 8), ((61, 59), 0.1, (2.0, 1.0), 0.05, 3),
                                                ((130, 65), 1.0, (0.0, 0.0), 1e-5, 32), ((2, 7), 1.0, (1.0, -0.5), 0.1, 2),
                                                ((33, 31, 29), 0.1, (1.0, -0.5, 0.3), 1e-3, 9),
                                                ((40, 37, 35), 0.1, (1.0, -1.0, 1.0), 0.1, 16)])
def test_refined_inverse_backward_error(sides, diff, vel, t, p, local):
    """The second correction starts from the first residual (r - tA d in float pairs) and both are added to
    x at once.  With u = 2^-53: the first residual carries at most 8 roundings of |tA||x|, the addition to
    x one, the pairs below 2^-40 of them and the third power of the FP32 inverse's error
    below all of it, so the residual in 64-bit-mantissa arithmetic stays under 16 u |tA||x| normwise."""
    need_gpu()
    from paper_1405_0707_gb300 import Plan
    n = int(np.prod(sides))
    V = inputs.rhs(n, p, 79)
    if local:
        V = np.zeros((n, p), order="F")
        V[np.linspace(0, n - 1, p).astype(int), np.arange(p)] = 1.0
    plan = Plan(sides, diff, vel, p_max=p, m=2, precision="mixed")
    W = to_np(plan.prec_apply(t, to_dev(V)))
    plan.close()
    A = sp.csr_matrix(ops.cd_matrix(sides, diff, vel, t))
    R = V.astype(np.longdouble) - _times_longdouble(A, W)
    scale = abs(A).sum(axis=1).max() * np.abs(W).max(axis=0)
    assert np.all(np.abs(R).max(axis=0) <= 16 * 2.0 ** -53 * scale)
