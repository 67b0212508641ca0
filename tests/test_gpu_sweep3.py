"""The one-launch 3D sweeps (small levels) against the half-sweep kernels, bit for
bit: a batch whose cells times sources pass the sweeps' limit of 131072 runs the
half sweeps, each of its sources alone the sweeps. Odd and even sides, a short
axis, levels that are not coarsened in every axis, all three cycle precisions."""
import numpy as np
import pytest

from gpu_util import fks, synth
from paper_1212_3660_gb300.solver import Solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [fks.FKS_PREC_MIXED, fks.FKS_PREC_MIXED_BF16])
@pytest.mark.parametrize("shape,mask", [((27, 25, 26), 63), ((64, 16, 17), 21), ((5, 60, 61), 42), ((40, 21, 22), 63),
                                        ((6, 7, 411), 63)])
def test_sweeps_equal_half_sweeps(shape, mask, precision):
    pr = synth.make_problem(shape, n_f=3, periods=(5.0, 3600.0), n_p=2, seed=39, dirichlet_mask=mask, n_src=8)
    assert pr.n <= 131072 < 8 * pr.n
    s = Solver(pr)
    b = pr.rhs().T.copy()
    kw = dict(precision=precision, inner_tol=1e-10, m_max=6, inner_max_cycles=3)
    batch = s.solve(b, **kw)
    assert np.isfinite(batch.X).all() and np.abs(batch.X).max() > 0
    for r in (0, 7):
        solo = s.solve(b[[r]], **kw)
        assert np.array_equal(solo.X[0], batch.X[r])
    s.close()
