"""The ACM step's lanes per node, chosen by size until a schedule is set: cells on both sides of a
line (64 nodes per SM in FP64, 448 in FP32) give the fields of the one-lane schedule.

Tolerance: only the order of the n_l = 25 term stencil sums differs, 25 eps of a sum's absolute terms,
which are at most ~100 times the fields' change per step; for 3 steps 3 x 25 x 100 eps = 7500 eps of the
largest value.
"""
import numpy as np
import pytest

import synth
from gpu_common import gpu_or_skip, rel_inf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n_axis", [("fp64", 21), ("fp64", 24), ("fp32", 40), ("fp32", 45)])
def test_default_lanes_equal_one_lane(prec, n_axis):
    rbf = gpu_or_skip()
    case = synth.jittered_cell(r=0.3, n_axis=n_axis, seed=4)
    s = rbf.Solver(0)
    s.set_case(case)
    s.build_stencils(25)
    s.compute_weights(solver=rbf.RBF_SOLVER_ACM)
    p, eps = (rbf.RBF_FP64, 2.0 ** -53) if prec == "fp64" else (rbf.RBF_FP32, 2.0 ** -24)
    got = []
    for code in (None, 256):
        if code:
            s.set_kernel_variant(code)
        s.init(precision=p, v_ref=0.01)
        s.step(3)
        got.append(s.get_fields())
    for c in range(4):
        assert np.abs(got[1][:, c]).max() > 0
        assert rel_inf(got[0][:, c], got[1][:, c]) <= 7500 * eps, c
    s.close()
