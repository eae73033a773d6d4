"""The FP32 inverse of the weight solve (PHS r^3, r^5) where it changes form: systems that just fill
and just pass a register tile (48, 64 unknowns), and the largest r^5 system (99 unknowns), in which
2 % of the stencils have a pivot below 1e-5 of its row and go on to the FP64 factors; against the FP64
oracle.

Tolerance: both sides solve their stored system to rounding, so they differ by what the rounding of
the stored matrix does, at most 2^-53 times the componentwise condition number (|M^-1| |M|, row sums)
per side; evaluated on the CPU for these stencils that number is at most 3.7e4 (r^3) and 6.4e6 (r^5):
1e-11 and 1.5e-9 in all.
"""
import pytest

import oracle
import synth
from gpu_common import gpu_or_skip, rowwise_rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cell():
    return synth.jittered_cell(r=0.3, n_axis=9, seed=7)


@pytest.mark.parametrize("n_l,m,k,tol", [(38, 2, 3, 1e-11), (39, 2, 3, 1e-11), (44, 3, 5, 1.5e-9), (50, 4, 5, 1.5e-9),
                                         (64, 4, 5, 1.5e-9)])
def test_acm_operators(cell, n_l, m, k, tol):
    rbf = gpu_or_skip()
    s = rbf.Solver(0)
    s.set_case(cell)
    s.build_stencils(n_l)
    assert s.compute_weights(k=k, m=m, solver=rbf.RBF_SOLVER_ACM)["n_singular"] == 0
    w = oracle.acm_weights(cell["xyz"], s.get_stencils(), k, m)
    for op in range(4):
        assert rowwise_rel(s.get_weights(op), w[:, op, :]) <= tol, op
    s.close()
