"""The bounded wait of the 3D coarse slab inverses: with a limit of zero iterations every thread block that waits for
another one's panel gives up, the factorisation returns FSI_E_TIMEOUT naming that wait (not the tensor core's), and the
same instance then factors and solves as before."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_1709_05660_gb300.workloads import Problem, SolverOpts, noise  # noqa: E402

E_TIMEOUT = -8


def _cut(a, b, n):
    return tuple(a + (b - a) * i / n for i in range(n + 1))


def test_wait_runs_out():
    from paper_1709_05660_gb300 import fsi
    prob = Problem(dim=3, breaks=(_cut(0.0, 1.0, 5), _cut(0.0, 0.5, 2), _cut(0.0, 0.5, 2)), levels=1,
                   flap_lo=(0.0, 0.0, 0.0), flap_hi=(0.34, 0.2, 0.5), mu_s=5e5, U=0.2)
    s = fsi.FSI(prob, SolverOpts(tile=(2, 2, 2)), stream=torch.cuda.current_stream().cuda_stream)
    try:
        n = int(s.N[-1])
        y = torch.empty(n, dtype=torch.float64, device="cuda")
        s.initial_state(torch.tensor(noise(n, 1), device="cuda"), y)
        s.set_state(y)
        s.assemble()
        b = torch.tensor(np.random.default_rng(3).standard_normal(n), device="cuda")
        z = [torch.empty_like(b), torch.empty_like(b)]
        s.factor()
        s.apply_vcycle(b, z[0])
        s.set_tc_wait_limit(0)
        with pytest.raises(fsi.FSIError) as ei:
            s.factor()
        assert ei.value.code == E_TIMEOUT and "slab" in str(ei.value)
        s.set_tc_wait_limit(-1)
        s.factor()
        s.apply_vcycle(b, z[1])
        assert torch.equal(z[0], z[1])
    finally:
        s.close()
