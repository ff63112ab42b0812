"""Mixed plans on grids with axes of one point, where strides of the exact inverse's transforms coincide."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import cf, operators as ops
from paper_1405_0707_gb300 import inputs
from tests.gpu_util import need_gpu, rel, to_dev, to_np
from tests.test_gpu_mma import _times_longdouble

pytestmark = pytest.mark.gpu

SIDES = [(1, 1, 9), (1, 1, 64), (1, 9, 1), (9, 1, 1), (1, 1, 1), (1, 5, 7), (5, 1, 7), (5, 7, 1), (17, 1, 33), (1, 12, 16),
         (16, 12, 1), (1, 9), (9, 1), (1, 1), (64, 1), (1, 64)]


@pytest.mark.parametrize("p", [1, 3])
@pytest.mark.parametrize("sides", SIDES)
def test_refined_inverse(sides, p):
    """Backward error of (tA)^{-1} V within 16 roundings of |tA||x| (the bound of full grids)."""
    need_gpu()
    from paper_1405_0707_gb300 import Plan
    n, vel, t = int(np.prod(sides)), (0.5, -0.3, 0.2)[:len(sides)], 0.01
    V = inputs.rhs(n, p, 3)
    plan = Plan(sides, 1.0, vel, p_max=p, m=2, precision="mixed")
    X = to_np(plan.prec_apply(t, to_dev(V)))
    plan.close()
    A = sp.csr_matrix(ops.cd_matrix(sides, 1.0, vel, t))
    R = V.astype(np.longdouble) - _times_longdouble(A, X)
    scale = abs(A).sum(axis=1).max() * np.abs(X).max(axis=0)
    assert np.all(np.abs(R).max(axis=0) <= 16 * 2.0 ** -53 * scale)


@pytest.mark.parametrize("sides", [(1, 1, 64), (1, 64, 1), (64, 1, 1), (1, 12, 16), (17, 1, 33)])
def test_solve(sides):
    need_gpu()
    from paper_1405_0707_gb300 import Plan
    n, vel, t = int(np.prod(sides)), (0.5, -0.3, 0.2), 0.01
    B = inputs.rhs(n, 2, 3)
    plan = Plan(sides, 1.0, vel, p_max=2, m=8, tol=1e-11, max_cycles=200, precision="mixed", algorithm=2)
    Z, info = plan.expm_block(t, to_dev(B))
    assert info.converged == 1
    ref = ops.exact_r_of_A_B(sides, 1.0, vel, t, cf.load_table(), B)
    assert rel(to_np(Z), ref) <= 1e-9 * np.linalg.norm(B) / np.linalg.norm(ref)
    plan.close()


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("sides,p", [((61, 59), 3), ((32, 24), 8), ((13, 12, 11), 5), ((16, 12, 20), 4)])
def test_unaligned_columns(sides, p, precision):
    """Columns that start 8 bytes past a 16-byte boundary, an odd number of rows apart: the same values, bit for
    bit, as with packed columns."""
    torch = need_gpu()
    from paper_1405_0707_gb300 import Plan
    n, vel, t = int(np.prod(sides)), (0.5, -0.3, 0.2)[:len(sides)], 0.01

    def odd():
        return torch.zeros((p, n + 3 + n % 2), dtype=torch.float64, device="cuda")[:, 1:n + 1].T

    B, X, Z, Xo, Zo = to_dev(inputs.rhs(n, p, 3)), None, None, odd(), odd()
    Bo = odd()
    Bo.copy_(B)
    plan = Plan(sides, 1.0, vel, p_max=p, m=6, fixed_cycles=2, precision=precision, algorithm=2)
    X, (Z, _) = plan.prec_apply(t, B), plan.expm_block(t, B)
    plan.prec_apply(t, Bo, Xo)
    plan.expm_block(t, Bo, Zo)
    assert np.array_equal(to_np(Xo), to_np(X)) and np.array_equal(to_np(Zo), to_np(Z))
    plan.close()
