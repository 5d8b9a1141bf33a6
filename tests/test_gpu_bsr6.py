"""The 3D operator's product (6 x 6 blocks, one warp per block row) against the exported matrix: block rows of few and
of many blocks, meshes whose block count is no multiple of a thread block's rows, the pressures' padded blocks, every
level.  Bar: the rounding bound of a sum of m products in any order, m eps (|A| |x|), m the longest row."""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_1709_05660_gb300.workloads import Problem, SolverOpts, noise  # noqa: E402


def _cut(a, b, n):
    return tuple(a + (b - a) * i / n for i in range(n + 1))


@pytest.mark.parametrize("nx,ny,nz,levels", [(1, 2, 2, 1), (2, 3, 1, 1), (3, 2, 2, 2), (5, 2, 3, 1)])
def test_operator_product(nx, ny, nz, levels):
    from paper_1709_05660_gb300 import fsi
    prob = Problem(dim=3, breaks=(_cut(0.0, 1.0, nx), _cut(0.0, 0.5, ny), _cut(0.0, 0.5, nz)), levels=levels,
                   flap_lo=(0.0, 0.0, 0.0), flap_hi=(0.34, 0.2, 0.5), mu_s=5e5, U=0.2)
    s = fsi.FSI(prob, SolverOpts(tile=(2, 2, 2)), stream=torch.cuda.current_stream().cuda_stream)
    try:
        n = int(s.N[levels - 1])
        y = torch.empty(n, dtype=torch.float64, device="cuda")
        s.initial_state(torch.tensor(noise(n, 1), device="cuda"), y)
        s.set_state(y)
        s.assemble()
        for lev in range(levels):
            rowptr, col, val = s.export_csr(lev)
            N = int(s.N[lev])
            A = sp.csr_matrix((val, col, rowptr), shape=(N, N))
            x = np.random.default_rng(5 + lev).standard_normal(N)
            out = torch.empty(N, dtype=torch.float64, device="cuda")
            s.apply_operator(lev, torch.tensor(x, device="cuda"), out)
            bar = np.diff(rowptr).max() * np.finfo(np.float64).eps * (abs(A) @ np.abs(x)) + np.finfo(np.float64).tiny
            assert np.all(np.abs(out.cpu().numpy() - A @ x) <= bar)
    finally:
        s.close()
