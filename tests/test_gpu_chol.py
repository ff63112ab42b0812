"""The FP64 Cholesky-QR's factor against the inverse that is applied (k_chol)."""
import numpy as np
import pytest

from paper_1405_0707_gb300 import inputs
from tests.gpu_util import need_gpu, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sides,count", [((31, 29), 300), ((401, 251), 40)])
def test_one_column_factor(sides, count):
    """p = 1, where R is a number: W = V_0 h + V_1 R up to a scale error of V_1 of at most one rounding for each of
    the two passes' reciprocals and one for the product of their roots (3 u, u = 2^-53); the roundings of the
    n entries average out against V_1 (a quarter of u)."""
    need_gpu()
    from paper_1405_0707_gb300 import Plan
    L = np.longdouble
    plan = Plan(sides, 0.1, (1.0, -0.5), p_max=1, m=2)
    worst = 0.0
    for seed in range(count):
        v = inputs.rhs(plan.n, 1, seed)
        V, H = plan.arnoldi(0.05, to_dev(v / np.linalg.norm(v)))
        W = to_np(plan.prec_apply(0.05, V[:, :1])).astype(L)[:, 0]
        V, H = to_np(V).astype(L), to_np(H).astype(L)
        r = W - V[:, 0] * H[0, 0] - V[:, 1] * H[1, 0]
        worst = max(worst, abs(float(V[:, 1] @ r / H[1, 0])))
    plan.close()
    assert worst <= 3.25 * 2.0 ** -53


@pytest.mark.parametrize("sides,p", [((300, 300), 4), ((300, 300), 8), ((401, 251), 1), ((1000, 900), 1), ((150, 150), 24),
                                     ((800, 700), 3), ((400, 400), 4), ((500, 400), 6)])
def test_norms_of_localised_columns(sides, p):
    """Columns of (tA)^{-1} applied to unit vectors: one large entry, all others small.  Their norms come from the
    Gram matrix of the FP64 kernels or, on large blocks of three or more columns, of the digit products; its
    partial sums and factor take about ten roundings."""
    need_gpu()
    from paper_1405_0707_gb300 import Plan
    plan = Plan(sides, 0.1, (1.0, -0.5), p_max=p, m=2)
    assert plan.n * p >= 100000
    V1 = np.zeros((plan.n, p), order="F")
    V1[np.linspace(0, plan.n - 1, p).astype(int), np.arange(p)] = 1.0
    V = to_np(plan.arnoldi(0.05, to_dev(V1))[0]).astype(np.longdouble)
    plan.close()
    assert np.max(np.abs((V * V).sum(axis=0) - 1.0)) <= 16 * 2.0 ** -53


@pytest.mark.parametrize("sides,p,m", [((800, 700), 3, 3), ((400, 400), 4, 4), ((706, 708), 3, 2), ((354, 353), 4, 3), ((500, 400), 2, 3)])
def test_relation_and_orthogonality_on_either_side_of_the_digit_passes(sides, p, m):
    """Three and four columns just below and well above the sizes from which FP64 plans take the digit passes, and two,
    which never do: the bounds of the FP64 kernels and of the digit passes (1e-13)."""
    need_gpu()
    from paper_1405_0707_gb300 import Plan
    plan = Plan(sides, 0.1, (1.0, -0.5), p_max=p, m=m)
    V1 = np.linalg.qr(inputs.rhs(plan.n, p, 8))[0]
    V, H = plan.arnoldi(0.05, to_dev(V1))
    W = np.column_stack([to_np(plan.prec_apply(0.05, V[:, j * p:(j + 1) * p])) for j in range(m)])
    V, H = to_np(V), to_np(H)
    plan.close()
    assert np.linalg.norm(W - V @ H) <= 1e-13 * np.linalg.norm(W)
    assert np.linalg.norm(V.T @ V - np.eye((m + 1) * p)) <= 1e-13
