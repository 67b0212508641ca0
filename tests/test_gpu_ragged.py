"""Fused 2D levels with odd sides: the last coarse cell has one child. The fused
tile kernels perform the per-sweep kernels' operations in the same order, so one
V-cycle is bitwise the same for every tiling, at sides around the tiles' edges."""
import numpy as np
import pytest

from gpu_util import fks, synth
from paper_1212_3660_gb300.solver import Solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [fks.FKS_PREC_FP64, fks.FKS_PREC_MIXED, fks.FKS_PREC_MIXED_BF16])
@pytest.mark.parametrize("shape,mask", [((33, 35), 15), ((65, 31), 15), ((47, 97), 5), ((129, 63), 15), ((64, 67), 10)])
def test_odd_sides_fused_bitwise(shape, mask, precision):
    pr = synth.make_problem(shape, n_f=4, periods=(5.0, 3600.0), n_p=1, seed=33, dirichlet_mask=mask)
    s = Solver(pr)
    rng = np.random.default_rng(6)
    v = rng.standard_normal(pr.n) + 1j * rng.standard_normal(pr.n)
    out = []
    for fuse, t16, t8 in ((0, 0, 0), (-1, 0, 0), (-1, -1, 0), (-1, -1, -1)):
        fks.fks_op_set_fusion(s.op, precision, fuse)
        fks.fks_op_set_tiles(s.op, precision, t16)
        fks.fks_op_set_tiles8(s.op, precision, t8)
        z = np.zeros(pr.n, np.complex128)
        fks.fks_precond_apply(s.op, 0.02j, v, z, 1e-10, cycles=2, precision=precision)
        out.append(z)
    s.close()
    assert np.isfinite(out[0]).all() and np.abs(out[0]).max() > 0
    for z in out[1:]:
        assert np.array_equal(out[0], z)
