"""A server batch reserves spare slots for requests that join it. The complex128
rules that choose kernels by the arithmetic of a launch (fused 2D levels, small
tiles) do not take its slots for sources: a served request of one source fuses
the levels that fks_solve fuses for it, and gives its bits."""
import numpy as np
import pytest

from paper_1212_3660_gb300 import fks, synth
from paper_1212_3660_gb300.solver import Solver

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu

EPS = 1e-10


def served(pr, precision, setup=lambda op: None):
    """The launches of one request of one source through a server."""
    s = Solver(pr)
    setup(s.op)
    opts, keep = fks.make_options(tol=pr.tol, m_max=pr.m_max, precision=precision, inner_tol=EPS, schedule=pr.schedule)
    r = fks.ServerRequest(s.op, pr.rhs().T.copy(), pr.sigma, pr.tau_bar, opts, keep, pr.n)
    srv = fks.fks_server_create(s.ctx, 8 << 30, lanes=1)
    fks.fks_server_submit(srv, r)
    assert fks.fks_server_wait(srv, r.ticket) == fks.FKS_OK
    launches = fks.fks_server_launches(srv)
    fks.fks_server_destroy(srv)
    alone = s.solve(precision=precision, inner_tol=EPS)
    s.close()
    assert np.array_equal(alone.X, r.X)
    return launches


# finest levels within the threshold of 393216 cells for one source and for four, not for 17
@pytest.mark.parametrize("shape", [(224, 224), (160, 150)])
def test_one_source_fuses_its_2d_levels(shape):
    need_gpu()
    pr = synth.make_problem(shape, n_f=5, periods=(5.0, 3600.0), n_p=3, seed=81, m_max=100)
    counted = served(pr, fks.FKS_PREC_FP64)
    # a threshold that was set counts the cells of a level, whatever the batch
    by_level = served(pr, fks.FKS_PREC_FP64, lambda op: fks.fks_op_set_fusion(op, fks.FKS_PREC_FP64, 393216))
    assert counted == by_level
