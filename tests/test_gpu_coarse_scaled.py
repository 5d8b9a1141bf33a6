"""The 2D and 3D coarse solves (one-level instances: the V-cycle is the coarse solve) held to the accuracy of the method
that they stand for.  They scale the rows by powers of two before they factor, and so does the reference here: row maxima
to [1, 2), explicit inverse by partial-pivot LU, applied to the scaled right-hand side.

Bar: the componentwise backward error max |b - A x| / (|A| |x| + |b|) at most ten times the reference's (the order of
elimination differs, the bound does not), or n eps where that is larger.
"""
import numpy as np
import pytest
import scipy.linalg as sla

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import solver as osolver  # noqa: E402
from oracle.mesh import initial_state  # noqa: E402
from paper_1709_05660_gb300.workloads import Problem, SolverOpts, noise  # noqa: E402
from test_gpu_coarse_merge import _problem  # noqa: E402


def _cut(a, b, n):
    return tuple(a + (b - a) * i / n for i in range(n + 1))


def _box(nx, ny, nz):
    return Problem(dim=3, breaks=(_cut(0.0, 1.0, nx), _cut(0.0, 0.5, ny), _cut(0.0, 0.5, nz)), levels=1,
                   flap_lo=(0.0, 0.0, 0.0), flap_hi=(0.34, 0.2, 0.5), mu_s=5e5, U=0.2)


def _order(lev):
    """Unknowns by x: nodes, and elements between their planes."""
    dim = lev.dim
    node = np.arange(lev.n_nodes).repeat(2 * dim) % lev.nodes_ax[0]
    layer = 2 * (np.arange(lev.n_elem).repeat(dim + 1) % lev.cells[0]) + 1
    return np.argsort(np.concatenate([node, layer]), kind="stable")


@pytest.mark.parametrize("cells", [(1, 2), (5, 4), (8, 7), (13, 5), (16, 4), (17, 6), (24, 2), (24, 6), (3, 2, 1),
                                   (5, 3, 2), (6, 1, 2), (7, 4, 3)])
def test_backward_error(cells):
    from paper_1709_05660_gb300 import fsi
    prob = _problem(*cells) if len(cells) == 2 else _box(*cells)
    opts = SolverOpts(tile=(2,) * len(cells))
    orc = osolver.Oracle(prob, opts)
    N = orc.fine.N
    y0 = initial_state(prob, orc.fine, noise(N, 1))
    s = fsi.FSI(prob, opts, stream=torch.cuda.current_stream().cuda_stream)
    try:
        s.set_state(torch.tensor(y0, device="cuda"))
        s.assemble()
        s.factor()
        b = np.random.default_rng(3).standard_normal(N)
        z = torch.empty(N, dtype=torch.float64, device="cuda")
        s.apply_vcycle(torch.tensor(b, device="cuda"), z)
        z = z.cpu().numpy()
    finally:
        s.close()
    orc.assemble(y0)
    order = _order(orc.levels_mesh[0])
    A = orc.ops[0].J.toarray()[np.ix_(order, order)]
    v, z = b[order], z[order]
    scale = 2.0 ** -np.floor(np.log2(np.abs(A).max(axis=1)))
    inv = sla.lu_solve(sla.lu_factor(A * scale[:, None]), np.eye(N))

    def backward_error(x):
        return np.max(np.abs(v - A @ x) / (np.abs(A) @ np.abs(x) + np.abs(v)))

    bar = max(10.0 * backward_error(inv @ (scale * v)), N * np.finfo(np.float64).eps)
    assert backward_error(z) <= bar, (backward_error(z), bar)
