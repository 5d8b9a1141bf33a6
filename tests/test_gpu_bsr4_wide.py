"""The FP64 operator product of large 2D levels (two threads per row from 160,000 rows on) and of the level below
(four), against the exported matrix.  Bar: m eps (|A| |x|), m the longest row: the rounding bound of a sum of m
products in any order."""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_1709_05660_gb300.workloads import CONFIGS, noise  # noqa: E402


@pytest.mark.parametrize("level", [3, 4])
def test_operator_product(level):
    from paper_1709_05660_gb300 import fsi
    prob, opts = CONFIGS["channel2d_l5"]
    s = fsi.FSI(prob, opts, stream=torch.cuda.current_stream().cuda_stream)
    try:
        n = int(s.N[-1])
        y = torch.empty(n, dtype=torch.float64, device="cuda")
        s.initial_state(torch.tensor(noise(n, 1), device="cuda"), y)
        s.set_state(y)
        s.assemble()
        rowptr, col, val = s.export_csr(level)
        N = int(s.N[level])
        A = sp.csr_matrix((val, col, rowptr), shape=(N, N))
        x = np.random.default_rng(5).standard_normal(N)
        out = torch.empty(N, dtype=torch.float64, device="cuda")
        s.apply_operator(level, torch.tensor(x, device="cuda"), out)
        bar = np.diff(rowptr).max() * np.finfo(np.float64).eps * (abs(A) @ np.abs(x)) + np.finfo(np.float64).tiny
        assert np.all(np.abs(out.cpu().numpy() - A @ x) <= bar)
    finally:
        s.close()
