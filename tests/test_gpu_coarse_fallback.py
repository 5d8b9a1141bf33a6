"""Coarse operators that the parallel coarse factorisations cannot take and the sequential ones can: a level-0 operator
with identity Dirichlet rows is imported in which one slab's own block is singular (or nearly so) while the operator is
well conditioned - row a of slab k holds delta on its diagonal and 1 at an unknown b of the plane before it, row b holds
1 at both, every other row is dominated by its diagonal or, for an element's pressures (which have none) and the
unknowns at its centre that they pair with, by a 2 x 2 block [1 1; 1 0].  The 2D merged inverse then falls back to the banded LU, the
two-sided 3D chain (a in its last slab, which it eliminates first from the right) to the one-sided one.

Bar: the normwise forward error bound of an explicit inverse by partial pivoting, 10 n eps cond(A).
"""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_1709_05660_gb300.workloads import Problem, SolverOpts, noise  # noqa: E402

EPS = np.finfo(np.float64).eps
CELLS = {2: (7, 4), 3: (5, 2, 2)}


def _cut(a, b, n):
    return tuple(a + (b - a) * i / n for i in range(n + 1))


def _instance(dim, levels, precision=0):
    from paper_1709_05660_gb300 import fsi
    if dim == 2:
        prob = Problem(breaks=(_cut(0.0, 0.5, 2) + _cut(0.55, 2.0, CELLS[2][0] - 3), _cut(0.0, 0.5, CELLS[2][1])),
                       levels=levels, mu_s=5e5, U=0.2)
    else:
        nx, ny, nz = CELLS[3]
        prob = Problem(dim=3, breaks=(_cut(0.0, 1.0, nx), _cut(0.0, 0.5, ny), _cut(0.0, 0.5, nz)), levels=levels,
                       flap_lo=(0.0, 0.0, 0.0), flap_hi=(0.34, 0.2, 0.5), mu_s=5e5, U=0.2)
    s = fsi.FSI(prob, SolverOpts(tile=(2,) * dim, precision=precision), stream=torch.cuda.current_stream().cuda_stream)
    n = int(s.N[-1])
    y = torch.empty(n, dtype=torch.float64, device="cuda")
    s.initial_state(torch.tensor(noise(n, 1), device="cuda"), y)
    s.set_state(y)
    s.assemble()
    return s


def _operator(s, dim, slab, delta):
    """Values of level 0's pattern, in export order, and the matrix; slab: the slab of row a."""
    cells = CELLS[dim]
    nodes = [2 * c + 1 for c in cells]
    n_nodes, n_elem = int(np.prod(nodes)), int(np.prod(cells))
    _, _, dirichlet, _ = s.export_dofmap(0, n_nodes, n_elem)
    rowptr, col, val = s.export_csr(0)
    n = len(rowptr) - 1
    row = np.repeat(np.arange(n), np.diff(rowptr))
    off = np.random.default_rng(11).uniform(-0.5, 0.5, len(col)) / np.diff(rowptr)[row]
    off[dirichlet[row] | dirichlet[col]] = 0.0
    val = np.where(row == col, 1.0, off)
    for e in range(n_elem):
        centre, stride, r = 0, 1, e
        for c, m in zip(cells, nodes):
            centre += (2 * (r % c) + 1) * stride
            r, stride = r // c, stride * m
        for k in range(dim + 1):
            p, u = n_nodes * 2 * dim + e * (dim + 1) + k, centre * 2 * dim + k
            val[((row == p) & (col == u)) | ((row == u) & (col == p))] = 1.0
    mid = sum((m // 2) * int(np.prod(nodes[:k])) for k, m in enumerate(nodes) if k > 0)   # inside every other plane
    a, b = ((mid + 2 * slab + 1) * 2 * dim + dim, (mid + 2 * slab) * 2 * dim + dim)       # first velocity component
    assert not dirichlet[a] and not dirichlet[b]
    for i, entries in ((a, {a: delta, b: 1.0}), (b, {a: 1.0, b: 1.0})):
        val[rowptr[i]:rowptr[i + 1]] = [entries.get(int(j), 0.0) for j in col[rowptr[i]:rowptr[i + 1]]]
    A = sp.csr_matrix((val, col, rowptr), shape=(n, n)).toarray()
    return val, A


def _check(x, A, b):
    want = np.linalg.solve(A, b)
    bar = 10.0 * len(b) * EPS * np.linalg.cond(A)
    err = np.linalg.norm(x - want) / np.linalg.norm(want)
    assert bar < 1e-10 and err <= bar, (err, bar)


def _solve(s, apply, b):
    x = torch.empty(len(b), dtype=torch.float64, device="cuda")
    apply(torch.tensor(b, device="cuda"), x)
    return x.cpu().numpy()


# (the last one: an error of 3e-7 in the probe's row, where sound inverses stay below 3e-8)
@pytest.mark.parametrize("dim,slab,delta", [(2, 1, 0.0), (2, 4, 0.0), (2, 6, 0.0), (3, 4, 0.0), (2, 1, 1e-12),
                                            (2, 4, 1e-12), (2, 6, 1e-12), (3, 4, 1e-12), (2, 6, 2e-11)])
def test_one_level(dim, slab, delta):
    s = _instance(dim, 1)
    try:
        b = np.random.default_rng(3).standard_normal(int(s.N[0]))
        s.factor()
        plain = _solve(s, s.apply_vcycle, b)   # also records the V-cycle of the usual factors
        val, A = _operator(s, dim, slab, delta)
        s.import_csr(0, val)
        s.factor()
        _check(_solve(s, s.apply_vcycle, b), A, b)
        s.assemble()                           # and back to the usual ones
        s.factor()
        assert np.array_equal(_solve(s, s.apply_vcycle, b), plain)
    finally:
        s.close()


@pytest.mark.parametrize("batched", [False, True])
def test_two_levels(batched):
    from paper_1709_05660_gb300 import fsi
    one, two = _instance(2, 2, 1), _instance(2, 2, 1)
    try:
        n = int(one.N[0])
        b = np.random.default_rng(3).standard_normal(n)
        two.factor()
        plain = _solve(two, two.coarse_solve_static, b)
        val, A = _operator(one, 2, 3, 0.0)
        one.import_csr(0, val)
        if batched:
            fsi.factor_batch([one, two])
        else:
            one.factor()
            two.factor()
        _check(_solve(one, one.coarse_solve_static, b), A, b)
        assert np.array_equal(_solve(two, two.coarse_solve_static, b), plain)
    finally:
        one.close()
        two.close()
