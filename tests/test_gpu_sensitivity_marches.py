"""The sensitivity kernel where a strip has several steps (the values carried from
step to step), where the last strip is shorter than the others, and where a
warp's 31 cells lie in a full and a short strip, against the oracle.
test_gpu_sensitivity_strips.py's calls are small enough for strips of one step."""
import numpy as np
import pytest

from oracle.sensitivity import sensitivities
from paper_1212_3660_gb300 import synth
from paper_1212_3660_gb300.solver import Solver

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def strip_len(shape, n_f):
    """The launcher's rule: 16 steps while that leaves eight blocks per SM, then strips of equal length."""
    up = lambda a, b: -(-a // b)
    nm, part = shape[0], int(np.prod(shape[1:]))
    n = 16
    while n > 1 and up(part * up(nm, n), 31 * 8) * n_f < 8 * 152:
        n //= 2
    return up(nm, up(nm, n))


@pytest.mark.parametrize("shape,n_f,n_m,length", [((37, 29), 600, 2, 2), ((37, 29), 1300, 1, 13),
                                                  ((61, 200), 304, 2, 16), ((23, 5, 4), 1300, 9, 12),
                                                  ((13, 9, 31), 500, 2, 7)])
def test_strips_of_several_steps_match_oracle(shape, n_f, n_m, length):
    """Random phasors: the sums have at most 28 roundings of terms that the
    field's contrast can cancel by less than 1e3, so 1e-12 of the largest entry."""
    need_gpu()
    assert strip_len(shape, n_f) == length and shape[0] % length
    pr = synth.make_problem(shape, n_f=n_f, periods=(5.0, 3600.0), n_p=2, seed=44)
    s = Solver(pr)
    rng = np.random.default_rng(11)
    phi = rng.standard_normal((n_f, pr.n)) + 1j * rng.standard_normal((n_f, pr.n))
    psi = rng.standard_normal((n_m, n_f, pr.n)) + 1j * rng.standard_normal((n_m, n_f, pr.n))
    jk, js = s.sensitivity(phi, psi)
    s.close()
    for m in range(n_m):
        for j in (0, 1, n_f // 2, n_f - 1):
            ok, os_ = sensitivities(pr.shape, pr.h, pr.cond, pr.ss, pr.dirichlet_mask, pr.sigma[j], phi[j], psi[m, j])
            assert np.max(np.abs(jk[m, j] - ok)) <= 1e-12 * np.max(np.abs(ok)), (m, j)
            assert np.max(np.abs(js[m, j] - os_)) <= 1e-12 * np.max(np.abs(os_)), (m, j)
