"""Set-up of systems of different sizes in two threads at once, each with its own context: a launch's
shared memory must not depend on what another thread asked for last.  Counts of errors, and the
weights of a call alone bit for bit.
"""
import threading

import numpy as np
import pytest

import synth
from gpu_common import gpu_or_skip

pytestmark = pytest.mark.gpu


def test_weight_solves_of_different_sizes():
    rbf = gpu_or_skip()
    case = synth.jittered_cell(r=0.3, n_axis=6, seed=9)
    sizes = [(64, 3, 4), (12, 3, 1), (64, 7, 4), (12, 7, 1)]  # FP32 inverse and FP64 factors, largest and small
    errors, out = [], [set() for _ in sizes]

    def work(i):
        n_l, k, m = sizes[i]
        try:
            s = rbf.Solver(0)
            s.set_case(case)
            s.build_stencils(n_l)
            for _ in range(200):
                s.compute_weights(k=k, m=m, solver=rbf.RBF_SOLVER_ACM)
            out[i].add(s.get_weights(rbf.RBF_OP_LAP).tobytes())
            s.close()
        except rbf.RbfError as e:
            errors.append((sizes[i], str(e)))

    for i in range(len(sizes)):  # alone
        s = rbf.Solver(0)
        s.set_case(case)
        s.build_stencils(sizes[i][0])
        s.compute_weights(k=sizes[i][1], m=sizes[i][2], solver=rbf.RBF_SOLVER_ACM)
        w = s.get_weights(rbf.RBF_OP_LAP)
        assert np.isfinite(w).all()
        out[i].add(w.tobytes())
        s.close()
    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(sizes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    assert all(len(o) == 1 for o in out)
