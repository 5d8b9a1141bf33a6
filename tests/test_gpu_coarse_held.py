"""Held factors of a one-level instance (the V-cycle is the coarse solve): after another state's assembly, or another
operator's import, without a new factorisation, the solve is still that of the factored operator.  Bar: bitwise the
vector of before (the factors, and with them every operation, are the same)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_1709_05660_gb300.workloads import Problem, SolverOpts, noise  # noqa: E402


def _cut(a, b, n):
    return tuple(a + (b - a) * i / n for i in range(n + 1))


PROBLEMS = {
    2: Problem(breaks=(_cut(0.0, 0.5, 2) + _cut(0.55, 2.0, 5), _cut(0.0, 0.5, 4)), levels=1, mu_s=5e5, U=0.2),
    3: Problem(dim=3, breaks=(_cut(0.0, 1.0, 5), _cut(0.0, 0.5, 3), _cut(0.0, 0.5, 2)), levels=1,
               flap_lo=(0.0, 0.0, 0.0), flap_hi=(0.34, 0.2, 0.5), mu_s=5e5, U=0.2),
}


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("dim", [2, 3])
def test_held_factors(dim, precision):
    from paper_1709_05660_gb300 import fsi
    prob = PROBLEMS[dim]
    s = fsi.FSI(prob, SolverOpts(tile=(2,) * dim, precision=precision), stream=torch.cuda.current_stream().cuda_stream)
    try:
        n = int(s.N[-1])
        y = torch.empty(n, dtype=torch.float64, device="cuda")
        b = torch.tensor(np.random.default_rng(3).standard_normal(n), device="cuda")

        def linearise(seed):
            s.initial_state(torch.tensor(noise(n, seed), device="cuda"), y)
            s.set_state(y)
            s.assemble()

        def solve():
            z = torch.empty(n, dtype=torch.float64, device="cuda")
            s.apply_vcycle(b, z)
            return z.cpu().numpy()

        linearise(1)
        s.factor()
        want = solve()
        linearise(2)
        assert np.array_equal(solve(), want)
        _, _, val = s.export_csr(0)
        s.import_csr(0, 3.0 * val)
        assert np.array_equal(solve(), want)
        linearise(2)
        s.factor()
        assert not np.array_equal(solve(), want)
    finally:
        s.close()
