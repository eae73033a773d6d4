"""The neighbour search at its edges, bit for bit against the oracle's brute-force stencils: one cell in
the grid, all distances tied (a lattice, its nodes in random order), very uneven density (the search has to
widen), the smallest and the largest stencil, coordinates on the period, and the wall nodes' fluid-only
stencils through the Neumann weights."""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import gpu_or_skip

pytestmark = pytest.mark.gpu


def _stencils(rbf, xyz, n_l):
    s = rbf.Solver(0)
    s.set_nodes(xyz, np.zeros(len(xyz), np.uint8))
    s.build_stencils(n_l)
    got = s.get_stencils()
    s.close()
    return got


@pytest.mark.parametrize("n,n_l", [(2, 2), (9, 9), (33, 32), (70, 64), (64, 33), (500, 40)])
def test_small_sets(n, n_l):
    rbf = gpu_or_skip()
    xyz = np.random.default_rng(n).random((n, 3))
    xyz[0] = 0.0
    xyz[-1] = 1.0 - 2.0**-53
    assert np.array_equal(_stencils(rbf, xyz, n_l), oracle.knn(xyz, xyz, n_l))


@pytest.mark.parametrize("n_axis,n_l", [(4, 27), (6, 33), (8, 64), (9, 7)])
def test_ties(n_axis, n_l):
    rbf = gpu_or_skip()
    xyz = synth.permute(synth.lattice(n_axis), 2)["xyz"]
    assert np.array_equal(_stencils(rbf, xyz, n_l), oracle.knn(xyz, xyz, n_l))


@pytest.mark.parametrize("n_l", [20, 45, 64])
def test_uneven_density(n_l):
    rbf = gpu_or_skip()
    rng = np.random.default_rng(3)
    xyz = np.concatenate([0.5 + 0.01 * rng.standard_normal((3000, 3)), rng.random((400, 3))]) % 1.0
    assert np.array_equal(_stencils(rbf, xyz, n_l), oracle.knn(xyz, xyz, n_l))


def test_wall_stencils_of_a_sparse_cell():
    """Dense wall, thinned fluid: the fluid-only search goes past the box its density estimate gives."""
    rbf = gpu_or_skip()
    case = synth.jittered_cell(r=0.3, n_axis=11, seed=4)
    wxyz, wn = synth.sphere_surface(np.full(3, 0.5), 0.3, 0.07)
    fluid = case["xyz"][case["type"] == 0]
    fluid = fluid[np.random.default_rng(1).random(len(fluid)) < 0.6]
    case["xyz"] = np.concatenate([wxyz, fluid])
    case["type"] = np.concatenate([np.ones(len(wxyz), np.uint8), np.zeros(len(fluid), np.uint8)])
    case["normal"] = np.concatenate([wn, np.zeros_like(fluid)])
    n_l = 30
    s = rbf.Solver(0)
    s.set_case(case)
    s.build_stencils(n_l)
    idx = oracle.knn(case["xyz"], case["xyz"], n_l)
    assert np.array_equal(s.get_stencils(), idx)
    rep = s.compute_weights(solver=rbf.RBF_SOLVER_ACM)
    # the wall stencils act in the wall pressure of a step
    dt = oracle.acm_dt(rep["h_min"], 1.0)
    w4 = oracle.acm_weights(case["xyz"], idx)
    _, idxb = oracle.neumann_stencils(case, n_l)
    wgb = oracle.neumann_weights(case, idxb)
    s.init(precision=rbf.RBF_FP64, dt=dt, v_ref=0.01)
    s.step(3)
    want, _ = oracle.acm_run(case, idx, w4, idxb, wgb, np.zeros((case.n, 4)), 3, dt=dt, v_ref=0.01)
    got = s.get_fields()
    wall = case["type"] == 1
    assert np.abs(got[wall, 3] - want[wall, 3]).max() <= 1e-9 * np.abs(want[wall, 3]).max()
    s.close()
