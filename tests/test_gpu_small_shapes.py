"""Kernels at the edges of their ranges, against the oracle on small meshes.

* Galerkin coarsening (1D interpolations in registers): meshes with one coarse cell in a direction, interface
  elements (three row kinds) and Dirichlet rows, 2D and 3D.  Bar: the rows within 1e-10 of their largest entry (as for
  the other Galerkin comparisons: sums of a few thousand products with cancellation).
* FP64 Schwarz inverses: blocks inverted in shared memory (up to 160 unknowns) and by panels of 16 and of 8, ragged
  last tiles, non-owned rows.  Bar: 10 n eps cond of the equilibrated blocks (both sides are backward stable).
* Arnoldi step: up to 32 basis vectors in one launch, beyond in several; one and two Gram-Schmidt passes.  Bar: the
  true residual at the solver's tolerance, plus the rounding of its evaluation, m eps (|J| |x|); iterations within 10%
  of the oracle's.
"""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import solver as osolver  # noqa: E402
from oracle.mesh import initial_state  # noqa: E402
from paper_1709_05660_gb300.workloads import Problem, SolverOpts, noise  # noqa: E402

EPS = np.finfo(np.float64).eps


def _cut(a, b, n):
    return tuple(a + (b - a) * i / n for i in range(n + 1))


def _problem(cells, levels):
    if len(cells) == 3:
        return Problem(dim=3, breaks=(_cut(0.0, 1.0, cells[0]), _cut(0.0, 0.5, cells[1]), _cut(0.0, 0.5, cells[2])),
                       levels=levels, flap_lo=(0.0, 0.0, 0.0), flap_hi=(0.34, 0.2, 0.5), mu_s=5e5, U=0.2)
    nx, ny = cells
    left, low = max(1, nx // 4), max(1, ny // 2)
    x = _cut(0.0, 0.5, left) + _cut(0.55, 2.0, nx - left - 1)
    y = _cut(0.0, 0.25, low) + _cut(0.25, 0.5, ny - low)[1:]
    return Problem(breaks=(x, y), levels=levels, mu_s=5e5, U=0.2)


def _pair(prob, opts):
    from paper_1709_05660_gb300 import fsi
    orc = osolver.Oracle(prob, opts)
    y0 = initial_state(prob, orc.fine, noise(orc.fine.N, 1))
    r, _ = orc.assemble(y0)
    s = fsi.FSI(prob, opts, stream=torch.cuda.current_stream().cuda_stream)
    s.set_state(torch.tensor(y0, device="cuda"))
    s.assemble()
    return s, orc, r


@pytest.mark.parametrize("cells,levels", [((3, 2), 3), ((5, 3), 2), ((13, 5), 2), ((1, 2, 2), 2), ((3, 2, 1), 2)])
def test_galerkin(cells, levels):
    prob = _problem(cells, levels)
    s, orc, _ = _pair(prob, SolverOpts(tile=(2,) * len(cells)))
    try:
        for lev in range(levels - 1):
            rowptr, col, val = s.export_csr(lev)
            n = len(rowptr) - 1
            want = orc.ops[lev].J.tocsr()
            diff = abs(sp.csr_matrix((val, col, rowptr), shape=(n, n)) - want).max(axis=1).toarray().ravel()
            rows = abs(want).max(axis=1).toarray().ravel()
            assert np.max(diff / np.where(rows == 0, 1.0, rows)) <= 1e-10
    finally:
        s.close()


def _cond(ops):
    worst, nmax = 0.0, 0
    J = ops.J.tocsr()
    for pt in ops.patches:
        B = J[pt.dofs][:, pt.dofs].toarray()
        B = B / np.abs(B).max(axis=1, keepdims=True)
        B = B / np.abs(B).max(axis=0, keepdims=True)
        worst, nmax = max(worst, np.linalg.cond(B)), max(nmax, len(pt.dofs))
    return worst, nmax


@pytest.mark.parametrize("cells,tile", [((5, 3), (1, 1)), ((5, 3), (2, 2)), ((13, 5), (3, 3)), ((5, 4), (4, 4)),
                                        ((5, 4), (6, 6)), ((3, 2, 1), (1, 1, 1)), ((3, 2, 1), (2, 2, 2))])
def test_schwarz_fp64(cells, tile):
    s, orc, _ = _pair(_problem(cells, 2), SolverOpts(tile=tile))
    try:
        orc.factor()
        s.factor()
        ops = orc.ops[1]
        cond, nmax = _cond(ops)
        n = ops.J.shape[0]
        rng = np.random.default_rng(5)
        b, x = rng.standard_normal(n), rng.standard_normal(n)
        want = x + SolverOpts().omega * osolver.ras_apply(ops, b - ops.J @ x)
        out = torch.empty(n, dtype=torch.float64, device="cuda")
        s.apply_smoother(1, torch.tensor(b, device="cuda"), torch.tensor(x, device="cuda"), out)
        err = np.linalg.norm(out.cpu().numpy() - want) / np.linalg.norm(want)
        assert err <= 10 * nmax * EPS * cond, (err, nmax, cond)
    finally:
        s.close()


@pytest.mark.parametrize("passes", [1, 2])
def test_arnoldi_long_restart(passes):
    opts = SolverOpts(tile=(1, 1), n_pre=1, n_post=1, omega=0.1, restart=50, rtol=1e-10, gs_passes=passes)
    s, orc, r = _pair(_problem((8, 7), 2), opts)
    try:
        orc.factor()
        s.factor()
        x = torch.zeros(len(r), dtype=torch.float64, device="cuda")
        st = s.solve(torch.tensor(-r, device="cuda"), x)
        _, sto = orc.solve(-r)
        assert sto.iters > 32 and abs(st.iters - sto.iters) <= max(1, int(0.1 * sto.iters)), (st.iters, sto.iters)
        x = x.cpu().numpy()
        rowptr, col, val = s.export_csr(1)
        J = sp.csr_matrix((val, col, rowptr), shape=(len(r), len(r)))
        slack = np.diff(J.indptr).max() * EPS * np.linalg.norm(abs(J) @ np.abs(x))
        assert np.linalg.norm(r + J @ x) <= opts.rtol * np.linalg.norm(r) + slack
    finally:
        s.close()
