"""The 2D coarse solve (one-level instance: the V-cycle is the coarse solve) over the coarse grids its merged
inverse takes: one slab, odd and even slab counts, the narrowest and widest planes, and one beyond the kernel's
shared memory (banded LU); and an imported operator whose Dirichlet rows are not identity rows, which is solved over
all unknowns by the banded LU.

Bar: the componentwise backward error of x = X b, max |b - A x| / (|A| |x| + |b|), at most ten times that of the
general method's inverse (partial-pivot LU of the same matrix in the same ordering, columns by triangular solves),
or n eps where that is smaller.  Rows and columns of these operators differ in scale by 1e12, so no fixed multiple of
eps bounds it: the LU inverse itself measures 1e-13 to 1e-6.
"""
import numpy as np
import pytest
import scipy.linalg as sla

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import solver as osolver  # noqa: E402
from oracle.mesh import initial_state  # noqa: E402
from paper_1709_05660_gb300.workloads import Problem, SolverOpts, noise  # noqa: E402


def _cut(a, b, n):
    return [a + (b - a) * i / n for i in range(n + 1)]


def _problem(nx, ny):
    x = _cut(0.0, 2.0, nx) if nx < 3 else _cut(0.0, 0.5, max(1, nx // 4)) + _cut(0.55, 2.0, nx - max(1, nx // 4) - 1)
    low = max(1, ny // 2)
    y = _cut(0.0, 0.25, low) + _cut(0.25, 0.5, max(1, ny - low))[1:]
    return Problem(breaks=(tuple(x), tuple(y)), levels=1, mu_s=5e5, U=0.2)


@pytest.mark.parametrize("nx,ny", [(1, 2), (2, 3), (3, 2), (5, 4), (8, 7), (13, 5), (16, 4), (17, 6), (24, 2), (6, 9)])
def test_coarse_solve_backward_error(nx, ny):
    from paper_1709_05660_gb300 import fsi
    prob = _problem(nx, ny)
    orc = osolver.Oracle(prob, SolverOpts())
    N = orc.fine.N
    y0 = initial_state(prob, orc.fine, noise(N, 1))
    s = fsi.FSI(prob, SolverOpts(), stream=torch.cuda.current_stream().cuda_stream)
    try:
        s.set_state(torch.tensor(y0, device="cuda"))
        s.assemble()
        s.factor()
        b = np.random.default_rng(3).standard_normal(N)
        z = torch.empty(N, dtype=torch.float64, device="cuda")
        s.apply_vcycle(torch.tensor(b, device="cuda"), z)
        z = z.cpu().numpy()
        rowptr, col, val = s.export_csr(0)
        i = int(np.nonzero(orc.fine.dir_mask)[0][0])
        val[rowptr[i] + np.searchsorted(col[rowptr[i]:rowptr[i + 1]], i)] = 2.0
        s.import_csr(0, val)
        s.factor()
        z_all = torch.empty(N, dtype=torch.float64, device="cuda")
        s.apply_vcycle(torch.tensor(b, device="cuda"), z_all)
        z_all = z_all.cpu().numpy()
        orc.assemble(y0)
        lev = orc.levels_mesh[0]
        node = np.arange(lev.n_nodes).repeat(4) % lev.nodes_ax[0]
        layer = 2 * (np.arange(lev.n_elem).repeat(3) % lev.cells[0]) + 1
        order = np.argsort(np.concatenate([node, layer]), kind="stable")
        A = orc.ops[0].J.toarray()[np.ix_(order, order)]
        v = b[order]
        lu = sla.lu_solve(sla.lu_factor(A), np.eye(N)) @ v

        A2 = A.copy()
        A2[order == i, order == i] = 2.0

        def backward_error(x, A=A):
            return np.max(np.abs(v - A @ x) / (np.abs(A) @ np.abs(x) + np.abs(v)))

        bar = max(10.0 * backward_error(lu), N * np.finfo(np.float64).eps)
        assert backward_error(z[order]) <= bar, (backward_error(z[order]), bar)
        assert backward_error(z_all[order], A2) <= bar, (backward_error(z_all[order], A2), bar)
    finally:
        s.close()
