"""The weight solve over its range of system sizes: single-row and two-node stencils, sizes around
the 32- and 64-row edges, and the largest system (64 nodes + 35 monomials), for 4 and for q - 1
operators, against the FP64 oracle.

Tolerance: both sides solve their stored system to rounding, so they differ by what the rounding of
the stored matrix does, at most 2^-53 times the componentwise condition number (|M^-1| |M|, row sums);
for these stencils that number is at most 5e5 (evaluated on the CPU), i.e. 5e-11 per side, 1e-10 in all.
"""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import gpu_or_skip, rowwise_rel

pytestmark = pytest.mark.gpu

SIZES = [(2, 0, 3), (5, 1, 3), (16, 2, 3), (17, 2, 9), (22, 2, 3), (33, 2, 5), (45, 3, 5), (48, 4, 3), (64, 2, 7),
         (64, 4, 3), (64, 4, 9)]


@pytest.fixture(scope="module")
def cell():
    return synth.jittered_cell(r=0.3, n_axis=9, seed=7)


@pytest.mark.parametrize("n_l,m,k", SIZES)
def test_acm_operators(cell, n_l, m, k):
    rbf = gpu_or_skip()
    s = rbf.Solver(0)
    s.set_case(cell)
    s.build_stencils(n_l)
    rep = s.compute_weights(k=k, m=m, solver=rbf.RBF_SOLVER_ACM)
    assert rep["n_singular"] == 0
    w = oracle.acm_weights(cell["xyz"], s.get_stencils(), k, m)
    for op in range(4):
        assert rowwise_rel(s.get_weights(op), w[:, op, :]) <= 1e-10, op


@pytest.mark.parametrize("q", [15, 19])
@pytest.mark.parametrize("n_l,m,k", [(5, 1, 3), (22, 2, 3), (33, 2, 5), (64, 4, 3)])
def test_lbm_operators(cell, n_l, m, k, q):
    rbf = gpu_or_skip()
    s = rbf.Solver(0)
    s.set_case(cell)
    s.build_stencils(n_l)
    s.compute_weights(k=k, m=m, solver=rbf.RBF_SOLVER_LBM, q=q, dx=0.05)
    w = oracle.lbm_weights(cell["xyz"], s.get_stencils(), q, 0.05, k, m)
    for j in range(1, q):
        assert rowwise_rel(s.get_weights(rbf.RBF_OP_LBM0 + j), w[:, j, :]) <= 1e-10, j
