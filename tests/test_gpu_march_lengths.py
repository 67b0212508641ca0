"""The marching complex128 stencil kernels (operator apply, defect, true residual)
where a thread takes several cells: two or four of them (twice that in the true
residual), the last chunk cut short by a side that they do not divide, against
the operator assembled in NumPy. test_gpu_march.py's grids are small enough that
every thread marches over one cell."""
import numpy as np
import pytest

import oracle
from gpu_util import fks, need_gpu, residual_floor, synth
from paper_1212_3660_gb300.solver import Solver

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


def march_len(shape):
    """The launcher's rule: four cells a thread while that leaves 5 blocks per SM, halved on smaller grids."""
    nx, ny, nz = (list(shape[::-1]) + [1])[:3]
    up = lambda a, b: -(-a // b)
    cols = up(nx, 32) * (up(ny, 8) if nz > 1 else 1)
    R = 4
    while R > 1 and cols * (up(nz, R) if nz > 1 else up(ny, 8 * R)) < 760:
        R //= 2
    return R


@pytest.mark.parametrize("shape,R", [((1001, 1027), 4), ((701, 1027), 2), ((99, 96, 97), 4), ((31, 90, 130), 2)])
def test_several_cells_a_thread(shape, R):
    need_gpu()
    assert march_len(shape) == R and shape[0] % R
    pr = synth.make_problem(shape, n_f=3, periods=(5.0, 3600.0), n_p=1, seed=37, ss_var=0.25, m_max=3)
    op = oracle.assemble(pr.shape, pr.h, pr.cond, pr.ss, pr.dirichlet_mask)
    rng = np.random.default_rng(8)
    s = Solver(pr)
    tau = 0.05j
    A = (op.K + tau * op.M).tocsr()
    # apply: a sum of at most seven products of coefficients that the two sides
    # form with a few roundings each, so 64 units in the last place of |A||x| per cell
    x = rng.standard_normal((2, pr.n)) + 1j * rng.standard_normal((2, pr.n))
    y = np.zeros_like(x)
    fks.fks_op_apply(s.op, tau, x, y, 2)
    for q in range(2):
        assert np.all(np.abs(y[q] - A @ x[q]) <= 64 * U * (abs(A) @ np.abs(x[q])))
    # defect: its norm after one cycle
    z = np.zeros(pr.n, np.complex128)
    _, _, pnorm = fks.fks_precond_apply(s.op, tau, x[0], z, 1e-10, cycles=1, precision=fks.FKS_PREC_MIXED)
    r = x[0] - A @ z
    assert abs(pnorm - np.linalg.norm(r)) <= 32 * U * np.linalg.norm(abs(A) @ np.abs(z)) + 1e-13 * np.linalg.norm(r)
    # true residuals of three steps' x_j, far from converged
    out = s.solve(inner_tol=1e-6)
    s.close()
    b = pr.rhs()[:, 0]
    X = out.X[0].T
    floor = residual_floor(op, b, pr.sigma, X)
    ref = [np.linalg.norm(b - op.K @ X[:, j] - sg * (op.M @ X[:, j])) / np.linalg.norm(b) for j, sg in enumerate(pr.sigma)]
    assert max(ref) > 1e-3  # (the shift that is the preconditioner's own is nearly solved)
    for j in range(len(ref)):
        assert abs(out.res_true[0, j] - ref[j]) <= floor[j] + 1e-12 * ref[j], j
