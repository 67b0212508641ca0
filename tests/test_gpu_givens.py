"""The Givens update on the first steps of a recurrence, where its chain of
rotations is empty (one step), a single rotation, and a few: the coefficients
that the four lanes of the chain hand to each other start from one shared value.
Every shift's least-squares (or square-system) residual and solution after
exactly m steps, against the oracle's dense solve of the explicit matrix."""
import numpy as np
import pytest

from gpu_util import fks, need_gpu, oracle_run, rel_err, replay_arrays, synth
from paper_1212_3660_gb300.solver import Solver

pytestmark = pytest.mark.gpu


# shift counts below, at and past the four warps of a block, and many blocks
@pytest.mark.parametrize("variant", ["fgmres", "ffom"])
@pytest.mark.parametrize("m,n_f", [(1, 1), (1, 5), (2, 4), (2, 130), (3, 3), (5, 130)])
def test_first_steps_match_oracle(m, n_f, variant):
    """The oracle's inner cycles are replayed, so both sides run the same
    operations in complex128: inner solves agree to rounding times the number of
    cycles, below 1e-10, and five steps' small least-squares problems add little."""
    need_gpu()
    pr = synth.make_problem((24, 20), n_f=n_f, periods=(5.0, 3600.0), n_p=2, seed=61, m_max=m, tol=1e-13)
    _, ref = oracle_run(pr, 1e-10, variant=variant)
    assert ref.steps == m and np.all(ref.m_j == m)
    rc, mj = replay_arrays(pr, [ref])
    s = Solver(pr)
    out = s.solve(inner_tol=1e-10, replay_cycles=rc, replay_mj=mj,
                  variant=fks.FKS_FFOM if variant == "ffom" else fks.FKS_FGMRES)
    s.close()
    assert np.array_equal(out.m_j[0], ref.m_j)
    assert np.allclose(out.res_est[0], ref.res_est, rtol=1e-8, atol=1e-10)
    for j in range(n_f):
        assert rel_err(out.X[0, j], ref.x[:, j]) <= 1e-8, j
