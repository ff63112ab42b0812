"""A plan's results do not depend on what its workspace held when it was allocated.

EXPM_FILL_BYTE makes plan creation fill every buffer with one byte: 0, 0x3F (FP64 4.8e-4, the size of a
basis entry), 0x41 (2.3e6, far above one) and 0xFF (NaN).  Every solve is deterministic, so the results
have to be the same bit for bit.  The row counts leave 1, 8 and 15 rows in the last 16-row tile and 1 to
31 in the columns' padding.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import operators as ops
from paper_1405_0707_gb300 import inputs
from tests.gpu_util import need_gpu, to_dev, to_np
from tests.test_gpu_mma import _times_longdouble

pytestmark = pytest.mark.gpu

FILLS = (0, 0x3F, 0x41, 0xFF)


def _plan(kind, **kw):
    from paper_1405_0707_gb300 import Plan
    if kind == "toeplitz":
        return Plan.toeplitz(inputs.toeplitz_column(20), 703, **kw), 0.9
    if kind == "csr":
        indptr, indices, data = inputs.sparse_stencil_matrix((11, 9, 7), seed=3)
        return Plan.csr((data, indices, indptr), **kw), 0.3
    return Plan(kind, 0.1, (1.0, -0.5, 0.3)[:len(kind)], **kw), 0.05


def _same(run, monkeypatch):
    out = []
    for fill in FILLS:
        monkeypatch.setenv("EXPM_FILL_BYTE", str(fill))
        out.append(run())
    assert all(np.all(np.isfinite(x)) for x in out[0])
    for other in out[1:]:
        for a, b in zip(out[0], other):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("kind,p,opts", [((41, 25), 3, {}), ((23, 24), 8, {}), ((53, 35), 16, {}), ((27, 13), 24, {}),
                                         ((13, 11, 9), 4, {}), ((7,), 1, {}), ((401, 251), 1, {}), ((97, 83), 13, {}),
                                         ((33, 29), 3, dict(k_defl=6)), ((33, 29), 6, dict(certify=True)),
                                         ("toeplitz", 3, {}), ("csr", 3, {})])
def test_solve_is_independent_of_the_workspace(kind, p, opts, precision, monkeypatch):
    need_gpu()

    def run():
        plan, t = _plan(kind, p_max=p, m=5, tol=1e-10, max_cycles=60, precision=precision, **opts)
        Z, info = plan.expm_block(t, to_dev(inputs.rhs(plan.n, p, 5)))
        plan.close()
        return to_np(Z), np.array(list(info.resid))

    _same(run, monkeypatch)


@pytest.mark.parametrize("sides,p,m", [((97, 83), 16, 6), ((41, 25), 3, 8), ((61, 59), 8, 10), ((130, 65), 32, 3)])
def test_arnoldi_is_independent_of_the_workspace(sides, p, m, monkeypatch):
    need_gpu()
    n = int(np.prod(sides))
    V1 = np.linalg.qr(inputs.rhs(n, p, 8))[0]

    def run():
        plan, t = _plan(sides, p_max=p, m=m, precision="mixed")
        V, H = plan.arnoldi(t, to_dev(V1))
        plan.close()
        return to_np(V), to_np(H)

    _same(run, monkeypatch)


def test_batch_runs_right_after_its_plans_are_made():
    """Plan creation returns with nothing of its own pending on the plan's stream: a batch graph, which runs
    on another stream, may follow at once."""
    torch = need_gpu()
    from paper_1405_0707_gb300 import Plan
    from paper_1405_0707_gb300.api import Batch
    probs = [((61, 59, 47), 8), ((45, 41, 39), 3), ((300, 301), 16)]
    Bs = [to_dev(inputs.rhs(int(np.prod(s)), p, 3)) for s, p in probs]
    streams = [torch.cuda.Stream() for _ in range(len(probs) + 1)]
    torch.cuda.synchronize()
    for _ in range(4):
        plans = [Plan(s, 1.0, (1.0, -1.0, 0.5)[:len(s)], p_max=p, m=5, fixed_cycles=2, precision="mixed", stream=q)
                 for (s, p), q in zip(probs, streams)]
        batch = Batch(plans, [1e-3] * len(probs), Bs, stream=streams[-1])
        first = [to_np(Z) for Z in batch.run()[0]]
        for a, Z in zip(first, batch.run()[0]):
            assert np.array_equal(a, to_np(Z))
        batch.close()
        for plan in plans:
            plan.close()


@pytest.mark.parametrize("value,bits", [(None, 49), ("1", 49), ("3", 44)])
@pytest.mark.parametrize("sides,p", [((61, 59), 3), ((33, 31, 29), 9), ((16, 12, 20), 4)])
def test_refined_inverse_under_each_stencil_switch(sides, p, value, bits, monkeypatch):
    """(tA)^{-1} V of mixed plans with the residual's stencil in FP64 (unset, "1") and in float pairs ("3"): backward
    error within 16 roundings of |tA||x|, or 16 times 2^-48 of it, with a workspace that starts as NaN."""
    need_gpu()
    from paper_1405_0707_gb300 import Plan
    monkeypatch.setenv("EXPM_FILL_BYTE", "255")
    if value is None:
        monkeypatch.delenv("EXPM_STENCIL_FP64", raising=False)
    else:
        monkeypatch.setenv("EXPM_STENCIL_FP64", value)
    n, vel, t = int(np.prod(sides)), (1.0, -0.5, 0.3)[:len(sides)], 0.05
    V = inputs.rhs(n, p, 79)
    plan = Plan(sides, 0.1, vel, p_max=p, m=2, precision="mixed")
    X = to_np(plan.prec_apply(t, to_dev(V)))
    plan.close()
    A = sp.csr_matrix(ops.cd_matrix(sides, 0.1, vel, t))
    R = V.astype(np.longdouble) - _times_longdouble(A, X)
    scale = abs(A).sum(axis=1).max() * np.abs(X).max(axis=0)
    assert np.all(np.abs(R).max(axis=0) <= 2.0 ** -bits * scale)
