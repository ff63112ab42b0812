"""Cycle graphs on the legacy default stream: a plan there launches a cycle directly the first time and
as a captured graph afterwards.  Both issue the same kernels on the same data, so a solve's result is
the same, bit for bit, on the first and on later calls, on the default stream and on the caller's own,
and with graphs disabled; with another time, width or a later call in between as well."""
import numpy as np
import pytest

from paper_1405_0707_gb300 import inputs
from tests.gpu_util import need_gpu, to_dev, to_np

pytestmark = pytest.mark.gpu


def _plan(kind, precision, algorithm, stream=None):
    from paper_1405_0707_gb300 import Plan
    kw = dict(p_max=3, m=4, tol=1e-9, max_cycles=60, precision=precision, algorithm=algorithm, stream=stream)
    if kind == "toeplitz":
        return Plan.toeplitz(inputs.toeplitz_column(20), 700, **kw), 0.9
    if kind == "csr":
        indptr, indices, data = inputs.sparse_stencil_matrix((11, 9, 7), seed=3)
        return Plan.csr((data, indices, indptr), **kw), 0.3
    sides = (33, 21) if kind == "grid2d" else (13, 11, 9)
    return Plan(sides, 0.1, (1.0, -0.5, 0.3)[:len(sides)], **kw), 0.05


@pytest.mark.parametrize("kind,precision,algorithm", [("grid2d", "mixed", 0), ("grid2d", "fp64", 2), ("grid3d", "mixed", 2),
                                                      ("toeplitz", "fp64", 1), ("csr", "mixed", 1), ("csr", "fp64", 2)])
def test_default_stream_graphs_repeat_the_direct_launches(kind, precision, algorithm, monkeypatch):
    torch = need_gpu()
    plan, t = _plan(kind, precision, algorithm)
    B, B2 = (to_dev(inputs.rhs(plan.n, p, 17 + p)) for p in (3, 2))
    out = [to_np(plan.expm_block(t, B)[0]) for _ in range(2)]
    other = [to_np(plan.expm_block(1.5 * t, B2)[0]) for _ in range(2)]
    out.append(to_np(plan.expm_block(t, B)[0]))
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    own, _ = _plan(kind, precision, algorithm, stream=s)
    out.append(to_np(own.expm_block(t, B)[0]))
    torch.cuda.synchronize()
    monkeypatch.setenv("EXPM_DISABLE_GRAPHS", "1")
    direct, _ = _plan(kind, precision, algorithm)
    out.append(to_np(direct.expm_block(t, B)[0]))
    for Z in out[1:]:
        assert np.array_equal(Z, out[0])
    assert np.array_equal(other[0], other[1])
    assert np.all(np.isfinite(out[0]))


@pytest.mark.parametrize("own_stream", [False, True])
def test_more_times_than_graphs_are_kept(own_stream):
    """A plan keeps the 16 graphs used last.  20 times, one solve of several cycles each: 16 graphs at the end, and a
    time that repeats has or gets one, whatever came before; results repeat bit for bit."""
    torch = need_gpu()
    from paper_1405_0707_gb300 import Plan, _native as N
    B = to_dev(inputs.rhs(33 * 21, 3, 17))
    stream = torch.cuda.Stream() if own_stream else None
    torch.cuda.synchronize()
    plan = Plan((33, 21), 0.1, (1.0, -0.5), p_max=3, m=4, tol=1e-9, max_cycles=60, precision="mixed", stream=stream)
    times = [0.05 * 1.01 ** k for k in range(20)]

    def solve(t):
        Z, info = plan.expm_block(t, B)
        assert info.cycles >= 3
        return to_np(Z)

    first = [solve(t) for t in times]
    held, captures = N.expm_plan_graph_stats(plan._h)
    assert (held, captures) == (16, 20)
    assert np.array_equal(solve(times[-1]), first[-1])
    assert N.expm_plan_graph_stats(plan._h) == (16, 20)          # kept
    assert np.array_equal(solve(times[0]), first[0])
    assert N.expm_plan_graph_stats(plan._h) == (16, 21)          # had gone, captured again
    assert np.array_equal(solve(times[0]), first[0])
    assert np.array_equal(solve(times[-1]), first[-1])
    assert N.expm_plan_graph_stats(plan._h) == (16, 21)
    plan.close()
