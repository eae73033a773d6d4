"""Which schedule the persistent ACM driver takes.

A share whose local nodes have no room in shared memory sends the solve to the streaming driver,
and that answer holds for its element size and lanes per node only.  The cell of 30,306 nodes
(N_L = 25, 152 SMs) was followed through the shares on the CPU: with one lane per node in FP64 the
largest share reaches 953 nodes and there is room for 828, with 2 / 4 / 8 lanes 854 / 834 / 817 of
1296 / 1472 / 1496, in FP32 there is room for 5656 and more.
"""
import numpy as np
import pytest

import synth
from gpu_common import gpu_or_skip

pytestmark = pytest.mark.gpu


def _solver(rbf, case, n_l=25):
    s = rbf.Solver(0)
    s.set_case(case)
    s.build_stencils(n_l)
    s.compute_weights(solver=rbf.RBF_SOLVER_ACM)
    return s


def test_share_without_room_is_remembered_by_lanes_and_precision():
    rbf = gpu_or_skip()
    s = _solver(rbf, synth.jittered_cell(r=0.35, n_axis=33, seed=8))
    s.init(precision=rbf.RBF_FP64, v_ref=0.01)
    with pytest.raises(rbf.RbfError):  # no launch yet
        s.persistent_info()
    s.permeability(32)  # the probes of solve()
    launches, fields = [], []
    for _ in range(2):
        s.init(precision=rbf.RBF_FP64, v_ref=0.01)
        a = s.launch_count()
        s.solve(4, 1e-300)
        launches.append(s.launch_count() - a)
        fields.append(s.get_fields())
        assert not s.persistent_info()["resident"]
    assert launches[0] == launches[1] + 1  # the first one found no room, the second did not try again
    assert np.array_equal(fields[0], fields[1])
    for lanes in (2, 4, 8):
        s.set_persistent_block(1000 * lanes + 128)
        s.solve(4, 1e-300)
        i = s.persistent_info()
        assert i["resident"] and i["lanes"] == lanes and i["threads"] == 256, lanes
    s.close()


def test_share_without_room_in_fp64_fits_in_fp32():
    rbf = gpu_or_skip()
    s = _solver(rbf, synth.jittered_cell(r=0.35, n_axis=33, seed=8))
    for prec, resident in ((rbf.RBF_FP64, 0), (rbf.RBF_FP32, 1), (rbf.RBF_FP32C, 1), (rbf.RBF_FP64, 0)):
        s.init(precision=prec, v_ref=0.01)
        s.solve(4, 1e-300)
        assert s.persistent_info()["resident"] == resident, prec
    s.close()


@pytest.mark.parametrize("n_axis,resident", [(6, 1), (14, 1), (29, 1), (32, 1), (36, 0)])
def test_resident_up_to_the_capacity(n_axis, resident):
    rbf = gpu_or_skip()
    s = _solver(rbf, synth.jittered_cell(r=0.35, n_axis=n_axis, seed=8))
    s.init(precision=rbf.RBF_FP64, v_ref=0.01)
    s.solve(4, 1e-300)
    assert s.persistent_info()["resident"] == resident
    s.close()


def test_streaming_blocks_per_sm():
    """Every lane count has the same warps on an SM: 32 in FP32, 24 in FP64."""
    rbf = gpu_or_skip()
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    s = _solver(rbf, synth.jittered_cell(r=0.35, n_axis=48, seed=8))  # 94k nodes: more units than warps from two lanes
    for prec, warps in ((rbf.RBF_FP64, 24), (rbf.RBF_FP32, 32)):
        s.init(precision=prec, v_ref=0.01)
        for code in (2256, 4256, 4128, 8128):
            s.set_persistent_block(code)
            s.solve(2, 1e-300)
            i = s.persistent_info()
            assert not i["resident"] and i["blocks"] * i["threads"] == sms * warps * 32, (prec, code)
    s.close()


@pytest.mark.parametrize("prec,n_cells,lanes", [("fp64", 24, 2), ("fp64", 28, 1), ("fp32", 24, 1), ("fp32c", 24, 1)])
def test_batch_default_lanes(prec, n_cells, lanes):
    """About 510 units a cell.  FP64 grids hold 3,648 warps: 24 cells leave a short round over (3.4 rounds) and take
    two lanes per node, 28 cells (3.9) one; FP32 always one.  The same fields from blocks of 32 threads."""
    rbf = gpu_or_skip()
    b = rbf.Batch(0)
    for i in range(n_cells):
        b.add_cell(synth.jittered_cell(r=0.3, n_axis=25 + i % 3, seed=40 + i), 20)
    b.build(3, 2)
    p = {"fp64": rbf.RBF_FP64, "fp32": rbf.RBF_FP32, "fp32c": rbf.RBF_FP32C}[prec]
    got = []
    for code in (None, 32 if lanes == 1 else 1000 * lanes + 32):
        if code:
            b.set_persistent_block(code)
        b.init(precision=p, v_ref=0.01)
        assert [r["steps"] for r in b.solve(6, 1e-300, check_every=3)] == [6] * n_cells
        i = b.cell(0).persistent_info()
        assert i["lanes"] == lanes and not i["resident"] and i["threads"] == (32 if code else 256 // lanes)
        got.append([b.cell(j).get_fields() for j in range(n_cells)])
    for x, y in zip(*got):
        assert np.abs(x).max() > 0 and np.array_equal(x, y)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_descriptor_copies_change_nothing(prec):
    """40 cells: blocks of 256 threads hold copies of the descriptors in shared memory (46 kB per SM), blocks of 64
    and 32 read them from global memory (150 kB and more)."""
    rbf = gpu_or_skip()
    b = rbf.Batch(0)
    for i in range(40):
        b.add_cell(synth.jittered_cell(r=0.3, n_axis=7 + i % 2, seed=60 + i), 20)
    b.build(3, 2)
    got = []
    for code in (256, 64, 32):
        b.init(precision=rbf.RBF_FP64 if prec == "fp64" else rbf.RBF_FP32, v_ref=0.01)
        b.set_persistent_block(code)
        assert [r["steps"] for r in b.solve(20, 1e-300, check_every=7)] == [20] * 40
        got.append([b.cell(j).get_fields() for j in range(40)])
    for j in range(40):
        assert np.abs(got[0][j]).max() > 0 and all(np.array_equal(g[j], got[0][j]) for g in got[1:]), j


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("n_axis,n_l", [(14, 25), (29, 24)])
def test_one_lane_solve_equals_the_step_kernels(prec, n_axis, n_l):
    """Codes of one lane per node: the same sums in the same order, so the same bits, with the wall nodes by four
    lanes each (the grid; the smaller cell on a cluster of 64 warps) and by one (1,295 of them on the cluster)."""
    rbf = gpu_or_skip()
    s = _solver(rbf, synth.jittered_cell(r=0.35, n_axis=n_axis, seed=5), n_l)
    got = []
    for code in (None, 256, -8):
        s.init(precision=rbf.RBF_FP64 if prec == "fp64" else rbf.RBF_FP32, v_ref=0.01)
        if code:
            s.set_persistent_block(code)
            s.solve(40, 1e-300)
        else:
            s.set_kernel_variant(256)
            s.step(40)
        got.append(s.get_fields())
    assert np.abs(got[0]).max() > 0 and all(np.array_equal(g, got[0]) for g in got[1:])
    s.close()


@pytest.mark.parametrize("prec,n_axis,lanes,threads", [("fp32", 34, 1, 512), ("fp32c", 34, 1, 512), ("fp64", 24, 2, 512)])
def test_tuner_times_the_schedule_by_size(prec, n_axis, lanes, threads):
    """Where no code names the schedule by size (512 threads, one lane resident) it is a candidate, code 0, so
    that tuning cannot lose it; setting 0 returns to it."""
    rbf = gpu_or_skip()
    s = _solver(rbf, synth.jittered_cell(r=0.35, n_axis=n_axis, seed=8))
    s.init(precision={"fp64": rbf.RBF_FP64, "fp32": rbf.RBF_FP32, "fp32c": rbf.RBF_FP32C}[prec], v_ref=0.01)
    want = dict(resident=1, cluster=0, threads=threads, lanes=lanes)
    s.solve(2, 1e-300)
    i = s.persistent_info()
    assert {k: i[k] for k in want} == want
    before = s.get_fields()
    times, chosen = s.autotune_persistent(100)
    assert np.array_equal(s.get_fields(), before)
    assert 0 in times and times[chosen] == min(times.values()) <= times[0]
    s.set_persistent_block(256)
    s.solve(2, 1e-300)
    assert not s.persistent_info()["resident"]
    s.set_persistent_block(0)
    s.solve(2, 1e-300)
    i = s.persistent_info()
    assert {k: i[k] for k in want} == want
    s.close()


def test_tuner_names_the_schedule_by_size_once():
    rbf = gpu_or_skip()
    s = _solver(rbf, synth.jittered_cell(r=0.35, n_axis=14, seed=5))  # by size: 256 threads, four lanes, as 4256
    s.init(precision=rbf.RBF_FP64, v_ref=0.01)
    assert 0 not in s.autotune_persistent(20)[0]
    s.close()
    b = rbf.Batch(0)
    for i in range(2):
        b.add_cell(synth.jittered_cell(r=0.3, n_axis=12, seed=70 + i), 20)
    b.build(3, 2)
    b.init(precision=rbf.RBF_FP32, v_ref=0.01)
    assert 0 not in b.autotune(20)[0]  # as 256


@pytest.mark.parametrize("prec,big", [("fp64", 1.7e308), ("fp32", 3.3e38)])
def test_wall_pressure_beyond_the_range(prec, big):
    """One fluid node's pressure near the largest value: a wall sum that overflows gives the same infinity in
    the resident driver as in the streaming one, and where it does not the same quotient (each sum has one
    term that counts: 4 eps)."""
    rbf = gpu_or_skip()
    case = synth.jittered_cell(r=0.35, n_axis=14, seed=5)
    s = _solver(rbf, case)
    wall = case["type"] == 1
    d = np.abs(np.linalg.norm(case["xyz"] - 0.5, axis=1) - 0.35)
    d[wall] = 1.0
    start = np.zeros((case.n, 4))
    start[d.argmin(), 3] = big
    p = []
    for code in (256, 4128):
        s.init(precision=rbf.RBF_FP64 if prec == "fp64" else rbf.RBF_FP32, v_ref=0.01, n_p=1)
        s.set_persistent_block(code)
        s.set_fields(start)
        with pytest.raises(rbf.RbfError) as ei:
            s.solve(1, 1e-300)
        assert ei.value.code == rbf.RBF_EDIVERGED
        assert s.persistent_info()["resident"] == (code == 4128)
        p.append(s.get_fields()[wall, 3])
    inf = np.isinf(p[0])
    assert inf.any() and (~inf & (np.abs(p[0]) > 1e-3 * big)).any() and not np.isnan(p[0]).any()
    assert np.array_equal(p[0][inf], p[1][inf])
    eps = 2.0 ** (-52 if prec == "fp64" else -23)
    x, y = p[0][~inf], p[1][~inf]
    assert (np.abs(x - y) <= 4 * eps * np.abs(x) + 1e-30 * big).all()
    s.close()
