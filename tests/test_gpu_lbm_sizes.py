"""The node-layout schedules of the lattice Boltzmann step over the sizes where their mapping changes
(8, 4, 2 lanes per node, one lane, the larger FP64 form, programmatic launches from 68k nodes),
against the FP64 oracle on ragged cells.  Tolerances as for the other schedules: FP64 populations 1e-9,
FP32 and refined FP32 1e-4 of the largest deviation from the rest weights.  The body force is large
(deviations far above rounding) for FP64 and FP32; the refined form is linearised about the rest state
and runs at the paper's scale, g = 1, as in its own parity test.
"""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import gpu_or_skip, rel_inf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_axis,q,n_l", [(9, 15, 21), (15, 19, 23), (19, 15, 20), (24, 19, 22), (30, 15, 25),
                                          (40, 15, 20), (46, 15, 20)])
def test_records_over_sizes(n_axis, q, n_l):
    rbf = gpu_or_skip()
    case = synth.jittered_cell(r=0.3, n_axis=n_axis, seed=11)
    assert case.n % 32
    dx, steps = 0.5 / n_axis, 6
    s = rbf.Solver(0)
    s.set_case(case)
    s.build_stencils(n_l)
    s.compute_weights(solver=rbf.RBF_SOLVER_LBM, q=q, dx=dx)
    idx = oracle.knn(case["xyz"], case["xyz"], n_l, grid=True)
    wk = oracle.lbm_weights(case["xyz"], idx, q, dx)
    tm = oracle.tau_minus(0.8, 3.0 / 16.0)
    f0 = oracle.lbm_equilibrium(q, np.ones(case.n), np.zeros((case.n, 3)))
    _, om, _ = oracle.velocity_set(q)
    for g, precs in (((2e4, 5e3, 0.0), ((rbf.RBF_FP64, 1e-9), (rbf.RBF_FP32, 1e-4))),
                     ((1.0, 0.0, 0.0), ((rbf.RBF_FP32R, 1e-4),))):
        u = oracle.lbm_units(1.0, 0.8, dx, g)
        fn = oracle.lbm_run(f0, q, case, idx, wk, 0.8, tm, u["g_lb"], steps)
        want = oracle.lbm_collide(fn, q, 0.8, tm, u["g_lb"])
        for prec, tol in precs:
            for code in (None, 6, 8, 9, 10):
                if code is not None:
                    s.set_kernel_variant(code)
                s.init(precision=prec, nu=1.0, g=g)
                s.step(steps)
                got = s.lbm_get_populations()
                assert rel_inf(got - om[:, None], want - om[:, None]) <= tol, (prec, code)
    s.close()
