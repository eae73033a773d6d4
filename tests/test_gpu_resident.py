"""The resident ACM driver (one cell, stencils in the SMs' shared memory) at the edges of its range,
against the FP64 oracle: fewer units than SMs, a ragged last unit, no wall nodes, cells near and past
the shared-memory capacity (the streaming driver takes over), more than one solve on one state.

Tolerances as for the other schedules: FP64 fields 1e-9, FP32 fields 1e-4 (both forms sum the same
terms in another order).
"""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import gpu_or_skip, oracle_acm_setup, rel_inf

pytestmark = pytest.mark.gpu


def _check(rbf, case, n_l, prec, tol, codes, steps=24, orc=None):
    o = orc or oracle_acm_setup(case, n_l)
    dt = oracle.acm_dt(o["h_min"], 1.0)
    rng = np.random.default_rng(3)
    start = 0.01 * rng.standard_normal((case.n, 4))
    start[case["type"] == 1, :3] = 0.0
    want, res = oracle.acm_run(case, o["idx"], o["w4"], o["idxb"], o["wgb"], start, steps, dt=dt, v_ref=0.01)
    s = rbf.Solver(0)
    s.set_case(case)
    s.build_stencils(n_l)
    s.compute_weights(solver=rbf.RBF_SOLVER_ACM)
    s.init(precision=prec, dt=dt, v_ref=0.01)
    for code in codes:
        if code:
            s.set_persistent_block(code)
        s.set_fields(start)
        # two solves in a row: the second starts from the first one's fields and max |v| slot
        assert s.solve(steps // 3, 1e-300, check_every=1)["steps"] == steps // 3
        r = s.solve(steps - steps // 3, 1e-300, check_every=100)
        assert r["steps"] == steps - steps // 3
        got = s.get_fields()
        for c in range(4):
            assert rel_inf(got[:, c], want[:, c]) <= tol, (code, c)
    s.close()


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-9), ("fp32", 1e-4), ("fp32c", 1e-4)])
@pytest.mark.parametrize("n_axis,n_l", [(5, 20), (8, 33), (14, 25)])
def test_small_cells(prec, tol, n_axis, n_l):
    rbf = gpu_or_skip()
    p = {"fp64": rbf.RBF_FP64, "fp32": rbf.RBF_FP32, "fp32c": rbf.RBF_FP32C}[prec]
    _check(rbf, synth.jittered_cell(r=0.3, n_axis=n_axis, seed=4), n_l, p, tol, (0, 2128, 4128, 8256))


def test_no_walls():
    rbf = gpu_or_skip()
    case = synth.lattice(8)
    rng = np.random.default_rng(5)
    case["xyz"] = (case["xyz"] + rng.uniform(-0.02, 0.02, case["xyz"].shape)) % 1.0
    _check(rbf, case, 20, rbf.RBF_FP64, 1e-9, (0, 4128))


@pytest.mark.parametrize("n_axis", [29, 34])  # about 20k and 33k nodes: inside and past the FP64 capacity
def test_capacity(n_axis):
    rbf = gpu_or_skip()
    _check(rbf, synth.jittered_cell(r=0.35, n_axis=n_axis, seed=8), 25, rbf.RBF_FP64, 1e-9, (0,), steps=9)
