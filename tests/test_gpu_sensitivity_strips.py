"""The sensitivity kernel's strips (fks_sensitivity) on narrow and odd grids:
rows and strips that begin and end inside a warp, a shorter last strip, more
measurements than one pass holds, against the oracle (oracle/sensitivity.py)."""
import numpy as np
import pytest

from oracle.sensitivity import sensitivities
from paper_1212_3660_gb300 import synth
from paper_1212_3660_gb300.solver import Solver

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


# (z,) y, x: strips of one step and longer (the shift count sets them), x sides
# below, at and above a warp's 31 cells
@pytest.mark.parametrize("shape,n_f,n_m", [((97, 3), 2, 9), ((37, 31), 90, 1), ((41, 64), 40, 2), ((35, 4, 5), 60, 1),
                                           ((19, 32, 33), 3, 1)])
def test_strips_match_oracle(shape, n_f, n_m):
    """Random phasors: the sums have at most 28 roundings of terms that the
    field's contrast can cancel by less than 1e3, so 1e-12 of the largest entry."""
    need_gpu()
    pr = synth.make_problem(shape, n_f=n_f, periods=(5.0, 3600.0), n_p=2, seed=43)
    s = Solver(pr)
    rng = np.random.default_rng(7)
    phi = rng.standard_normal((n_f, pr.n)) + 1j * rng.standard_normal((n_f, pr.n))
    psi = rng.standard_normal((n_m, n_f, pr.n)) + 1j * rng.standard_normal((n_m, n_f, pr.n))
    jk, js = s.sensitivity(phi, psi)
    for m in range(n_m):
        for j in range(0, n_f, max(1, n_f // 5)):
            ok, os_ = sensitivities(pr.shape, pr.h, pr.cond, pr.ss, pr.dirichlet_mask, pr.sigma[j], phi[j], psi[m, j])
            assert np.max(np.abs(jk[m, j] - ok)) <= 1e-12 * np.max(np.abs(ok)), (m, j)
            assert np.max(np.abs(js[m, j] - os_)) <= 1e-12 * np.max(np.abs(os_)), (m, j)
    s.close()
