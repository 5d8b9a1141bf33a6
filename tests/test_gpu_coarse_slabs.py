"""The 3D coarse solve from both ends of the slab chain (one-level instance: the V-cycle is the coarse solve): one to
six slabs (both parities, so the middle slab takes one correction or two), small and large planes, and slabs beyond
the kernel's row limit (one-sided chain).  Bar as in ``test_gpu_coarse_merge``: the componentwise backward error of
the solution at most ten times that of a partial-pivot LU inverse of the same matrix, or n eps."""
import numpy as np
import pytest
import scipy.linalg as sla

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import solver as osolver  # noqa: E402
from oracle.mesh import initial_state  # noqa: E402
from paper_1709_05660_gb300.workloads import Problem, SolverOpts, noise  # noqa: E402


def _cut(a, b, n):
    return tuple(a + (b - a) * i / n for i in range(n + 1))


@pytest.mark.parametrize("nx,ny,nz", [(1, 2, 2), (2, 2, 3), (3, 2, 1), (5, 3, 2), (6, 1, 2), (2, 6, 5)])
def test_coarse_slab_backward_error(nx, ny, nz):
    from paper_1709_05660_gb300 import fsi
    prob = Problem(dim=3, breaks=(_cut(0.0, 1.0, nx), _cut(0.0, 0.5, ny), _cut(0.0, 0.5, nz)), levels=1,
                   flap_lo=(0.0, 0.0, 0.0), flap_hi=(0.34, 0.2, 0.5), mu_s=5e5, U=0.2)
    orc = osolver.Oracle(prob, SolverOpts(tile=(2, 2, 2)))
    N = orc.fine.N
    y0 = initial_state(prob, orc.fine, noise(N, 1))
    s = fsi.FSI(prob, SolverOpts(tile=(2, 2, 2)), stream=torch.cuda.current_stream().cuda_stream)
    try:
        s.set_state(torch.tensor(y0, device="cuda"))
        s.assemble()
        s.factor()
        b = np.random.default_rng(3).standard_normal(N)
        z = torch.empty(N, dtype=torch.float64, device="cuda")
        s.apply_vcycle(torch.tensor(b, device="cuda"), z)
        z = z.cpu().numpy()
        orc.assemble(y0)
        A = orc.ops[0].J.toarray()
        lu = sla.lu_solve(sla.lu_factor(A), np.eye(N)) @ b

        def backward_error(x):
            return np.max(np.abs(b - A @ x) / (np.abs(A) @ np.abs(x) + np.abs(b)))

        bar = max(10.0 * backward_error(lu), N * np.finfo(np.float64).eps)
        assert backward_error(z) <= bar, (backward_error(z), bar)
    finally:
        s.close()
