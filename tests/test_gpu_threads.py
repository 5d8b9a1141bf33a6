"""Instances of different sizes factored by two host threads at once, each on its own stream: every launch takes its
own amount of shared memory from the same kernels, and neither thread's may limit the other's.  Results bitwise those
of each instance alone."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_1709_05660_gb300.workloads import Problem, SolverOpts, noise  # noqa: E402


def _cut(a, b, n):
    return tuple(a + (b - a) * i / n for i in range(n + 1))


def _box(ny, nz):
    return Problem(dim=3, breaks=(_cut(0.0, 1.0, 6), _cut(0.0, 0.5, ny), _cut(0.0, 0.5, nz)), levels=1,
                   flap_lo=(0.0, 0.0, 0.0), flap_hi=(0.34, 0.2, 0.5), mu_s=5e5, U=0.2)


CASES = {
    "fp64 blocks and merged inverse": [(Problem(levels=2), SolverOpts(tile=(1, 1))),
                                       (Problem(levels=2, breaks=(_cut(0.0, 0.5, 2) + _cut(0.55, 2.0, 5),
                                                                  _cut(0.0, 0.5, 6))), SolverOpts(tile=(2, 2)))],
    "mixed blocks": [(Problem(levels=2), SolverOpts(tile=(2, 2), precision=1)),
                     (Problem(levels=2), SolverOpts(tile=(4, 4), precision=1))],
    "slab chains": [(_box(2, 1), SolverOpts(tile=(2, 2, 2))), (_box(3, 3), SolverOpts(tile=(2, 2, 2)))],
}


@pytest.mark.parametrize("case", list(CASES))
def test_two_threads(case):
    from paper_1709_05660_gb300 import fsi
    streams = [torch.cuda.Stream() for _ in CASES[case]]
    inst, rhs, want = [], [], []
    for (prob, opts), st in zip(CASES[case], streams):
        s = fsi.FSI(prob, opts, stream=st.cuda_stream)
        n = int(s.N[-1])
        y = torch.empty(n, dtype=torch.float64, device="cuda")
        s.initial_state(torch.tensor(noise(n, 1), device="cuda"), y)
        s.set_state(y)
        s.assemble()
        s.factor()
        b = torch.tensor(np.random.default_rng(3).standard_normal(n), device="cuda")
        z = torch.empty_like(b)
        torch.cuda.synchronize()
        s.apply_vcycle(b, z)
        inst.append(s)
        rhs.append(b)
        want.append(z.cpu().numpy())
    errors = []

    def work(i):
        try:
            for _ in range(150):
                inst[i].factor()
        except Exception as e:   # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(inst))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for s, b, w in zip(inst, rhs, want):
        z = torch.empty_like(b)
        torch.cuda.synchronize()
        s.apply_vcycle(b, z)
        assert np.array_equal(z.cpu().numpy(), w)
        s.close()
