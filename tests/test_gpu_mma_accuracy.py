"""Accuracy of the mixed path's block step on blocks whose columns are localised (unit vectors), spread out, or
both: the cases where one row or one column dominates a product and the rest has to keep its own digits."""
import numpy as np
import pytest

from paper_1405_0707_gb300 import inputs
from tests.gpu_util import need_gpu, to_dev, to_np

pytestmark = pytest.mark.gpu

SHAPES = [((33, 31, 29), 9, 5), ((300, 300), 4, 10), ((97, 83), 16, 6), ((130, 65), 32, 4), ((64, 40), 17, 6),
          ((129, 127), 1, 12)]


def _start(kind, n, p):
    V1 = inputs.rhs(n, p, 8)
    if kind != "spread":
        first = 0 if kind == "local" else p // 2
        V1[:, first:] = 0.0
        V1[np.linspace(1, n - 2, p - first).astype(int), np.arange(first, p)] = 1.0
    return np.linalg.qr(V1)[0]


def _arnoldi(sides, p, m, V1):
    from paper_1405_0707_gb300 import Plan
    plan = Plan(sides, 0.1, (1.0, -0.5, 0.3)[:len(sides)], p_max=p, m=m, precision="mixed")
    V, H = plan.arnoldi(0.05, to_dev(V1))
    W = np.column_stack([to_np(plan.prec_apply(0.05, V[:, j * p:(j + 1) * p])) for j in range(m)])
    plan.close()
    return to_np(V), to_np(H), W


@pytest.mark.parametrize("kind", ["local", "half", "spread"])
@pytest.mark.parametrize("sides,p,m", SHAPES)
def test_relation(sides, p, m, kind):
    """(tA)^{-1} V_m = V_{m+1} H~_m.  V's digits resolve 2^-55 of a column's largest entry on each of the n <= 2^17
    rows (2^-46.5 of a unit column), the update's and the substitution's float pairs 2^-48 of the sums they
    hold, the FP32 correction V h2 2^-24 of an h2 near 2^-23 |W|: together below 2^-45 |W|."""
    need_gpu()
    V, H, W = _arnoldi(sides, p, m, _start(kind, int(np.prod(sides)), p))
    assert np.linalg.norm(W - V @ H) <= 2.0 ** -45 * np.linalg.norm(W)


@pytest.mark.parametrize("kind", ["local", "half", "spread"])
@pytest.mark.parametrize("sides,p,m", SHAPES)
def test_orthogonality(sides, p, m, kind):
    """The projections read V and W rounded to FP32 and add 16-row sums in float pairs: their error is that of
    the operands' rounding, 2^-24 of |V||W| entry by entry, whichever rows dominate."""
    need_gpu()
    V, _, _ = _arnoldi(sides, p, m, _start(kind, int(np.prod(sides)), p))
    assert np.abs(V.T @ V - np.eye((m + 1) * p)).max() <= 2.0 ** -24


@pytest.mark.parametrize("sides,p,m", [((90, 80, 70), 2, 10), ((90, 80, 70), 8, 10), ((600, 500), 17, 6), ((40, 41), 32, 12),
                                       ((33, 31), 17, 30), ((40, 41), 24, 19)])
def test_solution_columns_beside_localised_ones(sides, p, m):
    """Half of B's columns are unit vectors, half spread out, each of norm one; four cycles of Algorithm 1 converge
    far past FP64.  Against the FP64 plan, column by column: the coefficients of the solution update keep 2^-55
    of their largest scaled entry on n <= 2^19 rows and (m + 1) p columns (2^-43), and the partial fractions
    amplify the relation's 2^-48 by less than 2^6.  The last three shapes lie at and beyond the width up to which the digits
    fit in shared memory."""
    need_gpu()
    from paper_1405_0707_gb300 import Plan
    n, d = int(np.prod(sides)), len(sides)
    B = inputs.rhs(n, p, 4)
    B[:, p // 2:] = 0.0
    B[np.linspace(n // 3, n // 2, p - p // 2).astype(int), np.arange(p // 2, p)] = 1.0
    B /= np.linalg.norm(B, axis=0)
    t = 20.0 / sum((N + 1) ** 2 for N in sides)
    Z = []
    for precision in ("mixed", "fp64"):
        plan = Plan(sides, 0.1, (1.0, 1.0, 0.5)[:d], p_max=p, m=m, fixed_cycles=4, algorithm=1, precision=precision)
        Z.append(to_np(plan.expm_block(t, to_dev(B))[0]))
        plan.close()
    assert np.all(np.linalg.norm(Z[0] - Z[1], axis=0) <= 2.0 ** -41 * np.linalg.norm(Z[1], axis=0))
