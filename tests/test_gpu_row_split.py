"""The complex64 3D level kernels' cell addressing (rows split into j and k by a
multiplication, 32-bit indices) on sides where a row's division can go wrong:
one row per plane, one plane more than rows, odd and prime sides. One V-cycle of
the separate kernels equals, bit for bit, that of the tail kernel, which divides."""
import numpy as np
import pytest

from paper_1212_3660_gb300 import fks, synth
from paper_1212_3660_gb300.solver import Solver

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [fks.FKS_PREC_MIXED, fks.FKS_PREC_MIXED_BF16, fks.FKS_PREC_FP64])
@pytest.mark.parametrize("shape", [(16, 2, 16), (16, 1, 16), (2, 16, 16), (13, 7, 8), (8, 31, 2), (12, 10, 3)])
def test_level_kernels_equal_the_tail(shape, precision):
    need_gpu()
    pr = synth.make_problem(shape, n_f=4, periods=(5.0, 3600.0), n_p=1, seed=51)
    s = Solver(pr)
    rng = np.random.default_rng(9)
    v = rng.standard_normal(pr.n) + 1j * rng.standard_normal(pr.n)
    out = []
    for tail in (1, 1024):
        fks.fks_op_set_tail(s.op, precision, tail)
        z = np.zeros(pr.n, np.complex128)
        fks.fks_precond_apply(s.op, complex(pr.tau_bar[0]), v, z, 1e-10, cycles=2, precision=precision)
        out.append(z)
    s.close()
    assert np.isfinite(out[0]).all() and np.abs(out[0]).max() > 0
    assert np.array_equal(out[0], out[1])
