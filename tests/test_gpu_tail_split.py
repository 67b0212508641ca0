"""The tail in two launches around the coarsest product (complex128, a coarsest
level above 48 cells): bit for bit the per-level kernels' V-cycle, one level and
several, at 60 and 65 cells, for one source and for a batch; also
the cooperative lower cycle's, and the single-block tail's where pairs do not fit."""
import numpy as np
import pytest

from paper_1212_3660_gb300 import fks, synth
from paper_1212_3660_gb300.solver import Solver

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu

P = fks.FKS_PREC_FP64


@pytest.mark.parametrize("shape", [(9, 20, 14), (7, 20, 16), (13, 40), (16, 15), (8, 13, 20), (8, 42),
                                   (24, 21, 4)])
def test_split_tail_equals_level_kernels(shape):
    need_gpu()
    pr = synth.make_problem(shape, n_f=4, periods=(5.0, 3600.0), n_p=2, seed=53)
    s = Solver(pr)
    rng = np.random.default_rng(10)
    v = rng.standard_normal(pr.n) + 1j * rng.standard_normal(pr.n)
    b = rng.standard_normal((3, pr.n)) + 0j
    out = []
    for tail, coop in ((1, 0), (1024, 0), (4096, 0), (1, 1 << 30)):
        fks.fks_op_set_tail(s.op, P, tail)
        fks.fks_op_set_coop(s.op, P, coop)
        z = np.zeros(pr.n, np.complex128)
        fks.fks_precond_apply(s.op, complex(pr.tau_bar[0]), v, z, 1e-10, cycles=2, precision=P)
        x = s.solve(b=b, precision=P, inner_tol=1e-6).X
        out.append((z, np.asarray(x)))
    s.close()
    assert np.isfinite(out[0][0]).all() and np.abs(out[0][1]).max() > 0
    for other in out[1:]:
        for a, c in zip(out[0], other):
            assert np.array_equal(a, c)
