"""FP64 Schwarz blocks at the ends of the panel widths (16, 8 and 4 columns; the 4-column panel ends at 2,272
unknowns, above it the block is swept in device memory) against the oracle, and the cost of one block size beside the
next.  Bar of the smoother: 10 n eps cond of the equilibrated blocks (as in ``test_gpu_small_shapes``).
"""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import solver as osolver  # noqa: E402
from paper_1709_05660_gb300.workloads import SolverOpts  # noqa: E402
from test_gpu_small_shapes import EPS, _cond, _pair, _problem  # noqa: E402


@pytest.mark.parametrize("cells,levels,tile,lo,hi", [((8, 6), 2, (6, 11), 1380, 1461), ((8, 6), 2, (8, 9), 1462, 2200),
                                                     ((4, 3), 3, (12, 12), 2300, 2700)])
def test_schwarz_fp64_large(cells, levels, tile, lo, hi):
    s, orc, _ = _pair(_problem(cells, levels), SolverOpts(tile=tile))
    try:
        orc.factor()
        s.factor()
        assert lo < max(len(p.dofs) for p in orc.ops[levels - 1].patches) < hi
        for lev in range(1, levels):
            ops = orc.ops[lev]
            cond, nmax = _cond(ops)
            n = ops.J.shape[0]
            rng = np.random.default_rng(5)
            b, x = rng.standard_normal(n), rng.standard_normal(n)
            want = x + SolverOpts().omega * osolver.ras_apply(ops, b - ops.J @ x)
            out = torch.empty(n, dtype=torch.float64, device="cuda")
            s.apply_smoother(lev, torch.tensor(b, device="cuda"), torch.tensor(x, device="cuda"), out)
            err = np.linalg.norm(out.cpu().numpy() - want) / np.linalg.norm(want)
            assert err <= 10 * nmax * EPS * cond, (lev, err, nmax, cond)
    finally:
        s.close()


def test_cost_is_continuous():
    """Blocks of 1,394 unknowns (4-column panels) cost no more than four times those of 1,348 (8-column panels):
    twice the passes over a block, with as much again for noise.  The sweep in device memory takes ten and more."""
    def factor_s(tile):
        s, _, _ = _pair(_problem((8, 6), 2), SolverOpts(tile=tile))
        try:
            s.factor()
            best = 1e9
            for _ in range(3):
                t = time.perf_counter()
                s.factor()
                best = min(best, time.perf_counter() - t)
            return best
        finally:
            s.close()

    small, large = factor_s((8, 8)), factor_s((6, 11))
    assert large <= 4.0 * small, (small, large)
