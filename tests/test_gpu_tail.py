"""The single-block tail kernels against the per-level kernels, bit for bit: odd
sides, axes that are not coarsened, 2D and 3D, level sizes around the pair
kernel's 512 and 1024 pairs, several sources."""
import numpy as np
import pytest

from gpu_util import fks, synth
from paper_1212_3660_gb300.solver import Solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [fks.FKS_PREC_FP64, fks.FKS_PREC_MIXED])
@pytest.mark.parametrize("shape,mask", [((12, 10, 14), 63), ((14, 12, 13), 21), ((8, 16, 16), 63), ((6, 8, 20), 42),
                                        ((36, 37), 15), ((6, 90), 15), ((40, 26), 5), ((9, 12, 20), 63)])
def test_tail_thresholds_bitwise(shape, mask, precision):
    pr = synth.make_problem(shape, n_f=4, periods=(5.0, 3600.0), n_p=2, seed=37, dirichlet_mask=mask, n_src=2)
    s = Solver(pr)
    fks.fks_op_set_fusion(s.op, precision, 0)
    out = []
    for tail in (16, 64, 256, 1024, 4096):
        try:
            fks.fks_op_set_tail(s.op, precision, tail)
        except fks.FksError:
            continue  # f and z of that many cells do not fit in shared memory
        o = s.solve(precision=precision, inner_tol=1e-10, m_max=12, inner_max_cycles=3)
        out.append(o.X)
    s.close()
    assert len(out) >= 3 and np.isfinite(out[0]).all() and np.abs(out[0]).max() > 0
    for X in out[1:]:
        assert np.array_equal(out[0], X)
