"""Algorithmic bytes of the Arnoldi steps: up to 32 basis vectors one launch that reads the basis once more than it
makes Gram-Schmidt passes (the update of a pass shares its sweep with the products of the next), reads and writes w in
each pass, and reads it twice more while writing v_{j+1} once."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_1709_05660_gb300.workloads import Problem, SolverOpts, noise  # noqa: E402


@pytest.mark.parametrize("passes", [1, 2])
def test_krylov_bytes(passes):
    from paper_1709_05660_gb300 import fsi
    prob = Problem(levels=2)
    s = fsi.FSI(prob, SolverOpts(gs_passes=passes, restart=30), stream=torch.cuda.current_stream().cuda_stream)
    try:
        n = int(s.N[-1])
        y = torch.empty(n, dtype=torch.float64, device="cuda")
        s.initial_state(torch.tensor(noise(n, 1), device="cuda"), y)
        s.set_state(y)
        s.assemble()
        s.factor()
        s.set_profiling(True)
        _, st = s.newton_solve_update()
        stat = s.kernel_stats()["krylov"]
        nx, ny = (2 * (len(b) - 1) for b in prob.breaks)
        rows = 4 * ((2 * nx + 1) * (2 * ny + 1) + nx * ny)   # the padded layout's: four a node and a cell
        assert 1 < st.iters <= 30 and stat["launches"] == st.iters
        sweeps = sum((passes + 1) * (j + 1) + 2 * passes + 3 for j in range(st.iters))
        assert stat["bytes"] == 8 * rows * sweeps
    finally:
        s.close()
