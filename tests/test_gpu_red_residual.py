"""The restriction of the red cells' residual alone (complex128 cycles) against
the oracle's V-cycle (oracle/gmg.py), which restricts every cell's: two cycles
on hierarchies of every kind - halved in all axes, in some only, with odd sides,
one level - and every kernel that forms the residual."""
import numpy as np
import pytest

from oracle.gmg import Hierarchy
from paper_1212_3660_gb300 import fks, synth
from paper_1212_3660_gb300.solver import Solver

from gpu_util import need_gpu, oracle_op

pytestmark = pytest.mark.gpu

P = fks.FKS_PREC_FP64


@pytest.mark.parametrize("fuse,t16,t8,tail,cluster,coop", [(0, 0, 0, 64, 0, 0), (0, 0, 0, 64, 0, 1 << 30),
                                                           (-1, -1, 0, 64, 0, 0), (-1, -1, -1, 1024, 0, 0),
                                                           (-1, 0, 0, 64, 1024, 0)])
@pytest.mark.parametrize("shape", [(64, 64), (48, 23), (16, 12, 24), (9, 20, 14), (3, 30, 8), (4, 4)])
def test_two_cycles_match_oracle(shape, fuse, t16, t8, tail, cluster, coop):
    """The oracle's residual at a black cell is what rounding leaves of terms that
    cancel: a few 1e-16 of their size, which the smoother's contraction does not
    enlarge. Two cycles of at most 200 dependent roundings each, and a field
    whose contrast enlarges them by less than 100: 1e-11 of the largest entry."""
    need_gpu()
    pr = synth.make_problem(shape, n_f=4, periods=(5.0, 3600.0), n_p=1, seed=47)
    s = Solver(pr)
    fks.fks_op_set_fusion(s.op, P, fuse)
    fks.fks_op_set_tiles(s.op, P, t16)
    fks.fks_op_set_tiles8(s.op, P, t8)
    fks.fks_op_set_tail(s.op, P, tail)
    if cluster and shape == (64, 64):  # the cluster kernel wants levels halved in both axes
        fks.fks_op_set_cluster(s.op, P, cluster)
    fks.fks_op_set_coop(s.op, P, coop)
    rng = np.random.default_rng(8)
    v = rng.standard_normal(pr.n) + 1j * rng.standard_normal(pr.n)
    tau = complex(pr.tau_bar[0])
    z = np.zeros(pr.n, np.complex128)
    fks.fks_precond_apply(s.op, tau, v, z, 1e-10, cycles=2, precision=P)
    s.close()
    zo = Hierarchy(oracle_op(pr), [tau]).solve(v, 0, 1e-10, cycles=2)[0]
    assert np.max(np.abs(z - zo)) <= 1e-11 * np.max(np.abs(zo))
