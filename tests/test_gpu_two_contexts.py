"""Two contexts used by one thread each at the same time: the shared memory that
one operator's tail, coarsest product or cluster kernel may take is granted per
kernel and process, so the setup of the other operator, whose kernels need less,
must not take it away. Each apply gives the bits it gives alone."""
import threading

import numpy as np
import pytest

from gpu_util import fks, need_gpu, synth
from paper_1212_3660_gb300.solver import Solver

pytestmark = pytest.mark.gpu


def run(shapes, precision, tune, applies):
    probs = [synth.make_problem(sh, n_f=3, periods=(5.0, 3600.0), n_p=1, seed=71 + i) for i, sh in enumerate(shapes)]
    solvers = [Solver(p) for p in probs]
    for s in solvers:
        tune(s.op)
    rng = np.random.default_rng(5)
    vs = [rng.standard_normal(p.n) + 1j * rng.standard_normal(p.n) for p in probs]

    def apply(i):
        z = np.zeros(probs[i].n, np.complex128)
        fks.fks_precond_apply(solvers[i].op, complex(probs[i].tau_bar[0]), vs[i], z, 1e-10, cycles=6,
                              precision=precision)
        return z

    alone = [apply(i) for i in range(2)]
    wrong = []

    def loop(i):
        try:
            for _ in range(applies):
                if not np.array_equal(apply(i), alone[i]):
                    wrong.append((i, "other bits"))
        except fks.FksError as e:
            wrong.append((i, str(e)))

    threads = [threading.Thread(target=loop, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for s in solvers:
        s.close()
    assert not wrong, wrong[:4]


# the first operator's tail (1680 cells and below) needs more than the 48 KB that
# a kernel has without asking, the second's (144 cells) less
@pytest.mark.parametrize("precision", [fks.FKS_PREC_FP64, fks.FKS_PREC_MIXED])
def test_tails(precision):
    need_gpu()
    run([(37, 53, 45), (12, 12)], precision, lambda op: fks.fks_op_set_tail(op, precision, 2048), 60)


def test_clusters():
    need_gpu()
    run([(128, 128), (64, 64)], fks.FKS_PREC_MIXED, lambda op: fks.fks_op_set_cluster(op, fks.FKS_PREC_MIXED, 16384), 60)
