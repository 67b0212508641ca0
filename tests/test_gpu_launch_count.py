"""fks_profile_read counts every kernel launch, those of the coarsest inverse's
elimination among them: two in all for up to 40 unknowns, else one per step, or two
per step for many tiles, with one launch before and one after the steps."""
import numpy as np
import pytest

from gpu_util import fks, need_gpu, synth
from paper_1212_3660_gb300.solver import Solver

pytestmark = pytest.mark.gpu


def launches(shape):
    """Of one cycle on an operator of a single level (odd sides: never coarsened)."""
    pr = synth.make_problem(shape, n_f=3, periods=(5.0, 3600.0), n_p=1, seed=91)
    s = Solver(pr)
    z = np.zeros(pr.n, np.complex128)
    fks.fks_profile_read(s.op)
    fks.fks_precond_apply(s.op, complex(pr.tau_bar[0]), np.ones(pr.n, np.complex128), z, 1e-10, cycles=1)
    n = fks.fks_profile_read(s.op)["all_launches"]
    s.close()
    return n


@pytest.mark.parametrize("shape,steps", [((7, 9), 63), ((19, 19), 361), ((27, 27), 2 * 729)])
def test_elimination_steps_are_counted(shape, steps):
    need_gpu()
    assert launches(shape) - launches((5, 5)) == steps
