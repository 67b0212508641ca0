"""The coarsest level's inverse and its product: on a grid with a single
multigrid level one cycle is z = (K + tau M)^{-1} v, compared with a dense
NumPy solve. Sides are odd (or short), so the grid is not coarsened; the sizes
straddle the one-block inversion (up to 40 unknowns), the edges of the 32 x 32
tiles and the largest coarsest level; a negative tau makes the diagonal small,
so that rows are exchanged. Bound: a Gauss-Jordan inverse and one product have a
relative error of a modest multiple of n u kappa(A) (64 here), u the unit
roundoff of the cycle precision for the stored inverse and complex128's for the
elimination."""
import numpy as np
import pytest

import oracle
from gpu_util import fks, synth
from paper_1212_3660_gb300.solver import Solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [fks.FKS_PREC_FP64, fks.FKS_PREC_MIXED])
@pytest.mark.parametrize("kind", ["imaginary", "negative"])
@pytest.mark.parametrize("shape", [(3, 3), (4, 3), (5, 7), (3, 13), (1, 41), (7, 9), (5, 13), (3, 3, 7), (11, 9), (3, 5, 9),
                                   (31, 33)])
def test_single_level_inverse(shape, kind, precision):
    pr = synth.make_problem(shape, n_f=4, periods=(5.0, 3600.0), n_p=1, seed=31)
    op = oracle.assemble(pr.shape, pr.h, pr.cond, pr.ss, pr.dirichlet_mask)
    K, M = op.K.toarray(), np.diag(np.asarray(op.M.diagonal()))
    tau = 1j * 0.3 if kind == "imaginary" else -0.7 * np.median(np.diag(K) / np.diag(M)) + 0j
    A = K + tau * M
    s = Solver(pr)
    rng = np.random.default_rng(5)
    v = rng.standard_normal(pr.n) + 1j * rng.standard_normal(pr.n)
    z = np.zeros(pr.n, np.complex128)
    st, cycles, _ = fks.fks_precond_apply(s.op, tau, v, z, 1e-10, cycles=1, precision=precision)
    s.close()
    assert st == fks.FKS_OK and cycles == 1
    ref = np.linalg.solve(A, v)
    kappa = np.linalg.cond(A)
    u64, u = 2.0 ** -53, 2.0 ** -53 if precision == fks.FKS_PREC_FP64 else 2.0 ** -24
    # error in z: the inverse's (forward error u64 kappa), then the stored
    # inverse and its n products in the cycle precision, relative to |A^-1||v|
    bound = 64 * pr.n * kappa * u64 + (pr.n + 4) * u * np.linalg.norm(np.abs(np.linalg.inv(A)) @ np.abs(v)) / np.linalg.norm(ref)
    assert np.linalg.norm(z - ref) <= bound * np.linalg.norm(ref)
