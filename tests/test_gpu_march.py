"""The complex128 stencil kernels that march along z (3D) or y (2D): sides below,
at and past the 32 x 8 blocks and the march lengths, against the same operator
assembled in NumPy. Sums of at most seven products per cell: relative error of a
few units in the last place of |A||x| per cell, of sqrt-of-n sums for a norm."""
import numpy as np
import pytest

import oracle
from gpu_util import fks, synth
from paper_1212_3660_gb300.solver import Solver

pytestmark = pytest.mark.gpu

SHAPES = [(1, 9), (3, 33), (17, 31), (65, 97), (5, 7, 9), (3, 9, 33), (13, 8, 31), (9, 17, 65), (2, 40, 64), (41, 16, 32)]


def problem(shape):
    pr = synth.make_problem(shape, n_f=4, periods=(5.0, 3600.0), n_p=1, seed=35, ss_var=0.25)
    op = oracle.assemble(pr.shape, pr.h, pr.cond, pr.ss, pr.dirichlet_mask)
    rng = np.random.default_rng(7)
    return pr, op, rng


@pytest.mark.parametrize("shape", SHAPES)
def test_defect_norm(shape):
    pr, op, rng = problem(shape)
    v = rng.standard_normal(pr.n) + 1j * rng.standard_normal(pr.n)
    s = Solver(pr)
    z = np.zeros(pr.n, np.complex128)
    tau = 0.05j
    _, _, pnorm = fks.fks_precond_apply(s.op, tau, v, z, 1e-10, cycles=1, precision=fks.FKS_PREC_MIXED)
    s.close()
    A = op.matrix(tau) if hasattr(op, "matrix") else (op.K + tau * op.M).tocsr()
    r = v - A @ z
    floor = 32 * 2.0 ** -53 * np.linalg.norm(abs(A) @ np.abs(z))   # rounding of one residual
    assert abs(pnorm - np.linalg.norm(r)) <= floor + 1e-13 * np.linalg.norm(r)
