"""The complex64 3D level kernels (k_gs, k_gs_correct and the restriction, with
rows split into j and k by a multiplication and 32-bit indices) on sides where
the split can go wrong: one and two rows per plane, odd and prime sides. A level
above 131072 cells times sources runs them, each of its sources alone the
one-launch sweeps, which find their cells another way: the bits are the same.
(test_gpu_row_split.py's levels are all below that limit in complex64.)"""
import numpy as np
import pytest

from gpu_util import fks, need_gpu, synth
from paper_1212_3660_gb300.solver import Solver

pytestmark = pytest.mark.gpu

SWEEP_CELLS = 131072


@pytest.mark.parametrize("precision", [fks.FKS_PREC_MIXED, fks.FKS_PREC_MIXED_BF16])
@pytest.mark.parametrize("shape,n_src", [((260, 1, 257), 2), ((130, 1, 128), 8), ((181, 2, 183), 2), ((100, 2, 91), 8),
                                         ((97, 7, 98), 2), ((61, 7, 41), 8), ((47, 31, 46), 2), ((19, 31, 29), 8)])
def test_half_sweeps_equal_sweeps(shape, n_src, precision):
    need_gpu()
    pr = synth.make_problem(shape, n_f=3, periods=(5.0, 3600.0), n_p=2, seed=52)
    assert pr.n <= SWEEP_CELLS < n_src * pr.n
    s = Solver(pr)
    b = np.zeros((n_src, pr.n), np.complex128)  # a well each, in any cell (the thin grids have no inner ones)
    b[np.arange(n_src), np.random.default_rng(6).integers(0, pr.n, n_src)] = 1.0
    kw = dict(precision=precision, inner_tol=1e-10, m_max=4, inner_max_cycles=3)
    batch = s.solve(b, **kw)
    assert np.isfinite(batch.X).all() and np.abs(batch.X).max() > 0
    for r in (0, n_src - 1):
        solo = s.solve(b[[r]], **kw)
        assert np.array_equal(solo.X[0], batch.X[r])
    s.close()
