"""The LBM schedule until one is set, on both sides of its lines (nodes per SM): a pair of populations per warp
or node records.  The two sum the moments in different orders, so the fields' bits tell which one
ran: equal to the expected schedule's, not to the other's.
"""
import numpy as np
import pytest

import synth
from gpu_common import gpu_or_skip

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,q,per_sm,want", [
    ("fp32", 15, 60, 1), ("fp32", 15, 200, 10), ("fp32", 15, 480, 10), ("fp32", 15, 560, 1), ("fp32", 15, 1120, 1),
    ("fp32", 15, 1300, 10), ("fp32r", 15, 60, 1),
    ("fp32", 19, 50, 1), ("fp32", 19, 90, 10), ("fp64", 15, 33, 1), ("fp64", 15, 55, 10), ("fp64", 19, 22, 1),
    ("fp64", 19, 33, 10)])
def test_default_schedule(prec, q, per_sm, want):
    rbf = gpu_or_skip()
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n_axis = int(round((per_sm * sms / 0.9) ** (1.0 / 3.0)))
    case = synth.jittered_cell(r=0.3, n_axis=n_axis, seed=3)
    assert abs(case.n / sms - per_sm) < 0.12 * per_sm
    s = rbf.Solver(0)
    s.set_case(case)
    s.build_stencils(20)
    s.compute_weights(solver=rbf.RBF_SOLVER_LBM, q=q, dx=0.5 / n_axis)
    p = {"fp64": rbf.RBF_FP64, "fp32": rbf.RBF_FP32, "fp32r": rbf.RBF_FP32R}[prec]
    got = {}
    for code in (None, 1, 10):
        if code is not None:
            s.set_kernel_variant(code)
        s.init(precision=p, tau_plus=0.8, magic=3.0 / 16.0)
        s.step(20)
        got[code] = s.get_fields()
    assert np.abs(got[None]).max() > 0 and np.array_equal(got[None], got[want])
    assert not np.array_equal(got[1], got[10])
    s.close()
