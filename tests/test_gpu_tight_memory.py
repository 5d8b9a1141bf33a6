"""A server budget one byte below an FP64 instance's planned size: the instance is built with one workspace region for
the Schwarz blocks of all its levels, which are then factored level by level.  It stays within the budget and its
Newton steps are bitwise those of the unlimited server (the blocks of every level take the same kernel here)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_1709_05660_gb300.workloads import Problem, SolverOpts, noise  # noqa: E402

STEPS = 2


def _steps(budget, cancel_first=False):
    from paper_1709_05660_gb300 import fsi
    prob, opts = Problem(levels=4), SolverOpts(tile=(2, 2), precision=0)
    plan = fsi.FSI(prob, opts, plan_only=True)
    n, planned = int(plan.N[-1]), plan.hbm_bytes
    plan.close()
    srv = fsi.Server(hbm_budget_bytes=budget(planned), max_slots=1)
    try:
        tickets = [srv.submit(1, prob, opts, noise=noise(n, 1) if k == 0 else None, last=False, keep_dx=True)
                   for k in range(STEPS)]
        srv.drain()
        held = srv.resident_bytes()
        out = []
        for t in tickets:
            dx = np.empty(n)
            res = srv.poll(t, dx)
            assert res is not None and res["status"] == 0, res
            out.append(dx)
        return out, held, planned
    finally:
        srv.close()


def test_budget_below_the_planned_size():
    want, held, planned = _steps(lambda p: 0)
    got, held_tight, _ = _steps(lambda p: p - 1)
    assert held_tight < planned <= 1.02 * held and held_tight < held
    for a, b in zip(got, want):
        assert np.array_equal(a, b)


def test_budget_far_below_is_refused():
    from paper_1709_05660_gb300 import fsi
    with pytest.raises(fsi.FSIError):
        _steps(lambda p: p // 2)
