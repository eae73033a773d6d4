"""The measured work of the framework: what a program that uses it calls, at the sizes it meets.

Twelve listed cases and a sampler of more of the same ranges.  They stand for the four things a
user does: set a geometry up (stencils, weights), step or solve it with either solver in each
precision, read permeability and drag from it, and train and use the warm-start network.  Node
clouds are periodic unit cells with one sphere, refined towards its surface like the cells of
``bench.py``: a lattice of coarse cells, each divided 1..s times per axis by its wall distance,
one jittered node per part, and a Fibonacci set on the sphere.

Fields of a run whose state is held in FP32 come back as FP32 arrays, those of an FP64 run as
FP64, so that each output has the type it was computed in.
"""
import math
import random

import numpy as np
import torch

import paper_2404_14195_gb300 as rbf
from paper_2404_14195_gb300 import warmstart

PREC = {"fp64": rbf.RBF_FP64, "fp32": rbf.RBF_FP32, "fp32c": rbf.RBF_FP32C, "fp32r": rbf.RBF_FP32R}
NU, G, V_REF, TAU, MAGIC, M_P = 1.0, (1.0, 0.0, 0.0), 2.0, 0.8, 3.0 / 16.0, 32


# ---- node clouds ------------------------------------------------------------------------------

def _cloud(cells, levels, ramp, r, seed):
    """(xyz, type, normal, centre, radius): `cells` coarse cells per axis, divided `levels` times per
    axis at the wall, falling linearly to one part at the distance `ramp` from it."""
    rng = np.random.default_rng(seed)
    h = 1.0 / cells
    g = (np.arange(cells) + 0.5) * h
    mid = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    d = np.sqrt(((mid - 0.5) ** 2).sum(1)) - r
    want = h * (1.0 / levels + (1.0 - 1.0 / levels) * np.clip(d / ramp, 0.0, 1.0))
    parts = np.clip(np.rint(h / want), 1, levels).astype(int)
    out = []
    for s in range(1, levels + 1):
        m = mid[parts == s]
        if not len(m):
            continue
        hs = h / s
        o = ((np.arange(s) + 0.5) / s - 0.5) * h
        p = (m[:, None, :] + np.stack(np.meshgrid(o, o, o, indexing="ij"), -1).reshape(1, -1, 3)).reshape(-1, 3)
        p = p[np.sqrt(((p - 0.5) ** 2).sum(1)) - r >= 0.7 * hs]  # before the jitter: the same number for every seed
        out.append(p + rng.uniform(-0.2 * hs, 0.2 * hs, p.shape))
    fluid = np.concatenate(out)
    hw = h / levels
    nw = max(16, int(round(4.0 * math.pi * r * r / (hw * hw))))
    i = np.arange(nw) + 0.5
    z, a = 1.0 - 2.0 * i / nw, math.pi * (1.0 + math.sqrt(5.0)) * i + rng.uniform(0.0, 2.0 * math.pi)
    q = np.sqrt(1.0 - z * z)
    normal = np.stack([q * np.cos(a), q * np.sin(a), z], 1)
    normal /= np.sqrt((normal ** 2).sum(1))[:, None]
    wall = 0.5 + r * normal
    xyz = np.concatenate([wall, np.clip(fluid, 0.0, np.nextafter(1.0, 0.0))])
    typ = np.concatenate([np.ones(len(wall), np.uint8), np.zeros(len(fluid), np.uint8)])
    nrm = np.concatenate([normal, np.zeros_like(fluid)])
    return dict(xyz=np.ascontiguousarray(xyz), type=typ, normal=nrm, centre=np.full(3, 0.5), radius=float(r), h_min=hw)


def _case_cloud(c, seed):
    return _cloud(c["cells"], c["levels"], c["ramp"], c["r"], seed)


def _batch_cells(c):
    """The cells of a batch (plain values each): radii, refinement and stencil sizes vary over the batch."""
    rng = random.Random(c["layout"])
    return [dict(cells=rng.randint(c["cells_lo"], c["cells_hi"]), levels=rng.randint(2, 4), ramp=0.2,
                 r=rng.uniform(0.15, 0.48), n_l=rng.randint(20, 45)) for _ in range(c["n_cells"])]


def _start_fields(cloud, seed):
    """A smooth (u, v, w, p) start of the size of the steady flow, zero velocity on the wall: what a
    previous solve, a neighbouring cell or the network gives."""
    rng = np.random.default_rng(seed + 1000)
    x = cloud["xyz"]
    d = np.sqrt(((x - 0.5) ** 2).sum(1)) - cloud["radius"]
    shape = np.where(cloud["type"] == 1, 0.0, 1.0 - np.exp(-np.clip(d, 0.0, None) / 0.1))
    f = np.empty((len(x), 4))
    for j in range(4):
        a, ph, n = rng.uniform(0.2, 1.0), rng.uniform(0.0, 2.0 * math.pi, 3), rng.integers(1, 3, 3)
        wave = np.prod(np.cos(2.0 * math.pi * n * x + ph), 1)
        f[:, j] = a * wave if j == 3 else 0.02 * shape * ((1.0 if j == 0 else 0.0) + 0.3 * a * wave)
    return f


# ---- velocity sets (odd k listed, the even k after it opposite) ----------------------------------

_E15 = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 1), (1, 1, -1), (1, -1, 1), (1, -1, -1)]
_E19 = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)]


def _velocities(q):
    e = [(0, 0, 0)]
    for v in (_E15 if q == 15 else _E19):
        e += [v, tuple(-a for a in v)]
    e = np.array(e, np.float64)
    n1 = np.abs(e).sum(1)
    w = (np.where(n1 == 0, 2 / 9, np.where(n1 == 1, 1 / 9, 1 / 72)) if q == 15
         else np.where(n1 == 0, 1 / 3, np.where(n1 == 1, 1 / 18, 1 / 36)))
    return e, w


def _lbm_units(dx):
    dt = (TAU - 0.5) / 3.0 * dx * dx / NU
    return dt, np.array(G) * dt * dt / dx


def _start_populations(cloud, q, dx, seed):
    """Equilibrium of the smooth start in lattice units, (q, n)."""
    f = _start_fields(cloud, seed)
    dt, _ = _lbm_units(dx)
    v, rho = f[:, :3] * dt / dx, 1.0 + 1e-6 * f[:, 3]
    e, w = _velocities(q)
    eu = e @ v.T
    return w[:, None] * rho * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * (v * v).sum(1))


# ---- the cases -----------------------------------------------------------------------------------

def listed():
    return [
        # A new geometry of the size of a quick study (7k nodes, N_L = 25, PHS r^3, m = 2): order the nodes, find
        # the stencils, solve the weights and read them, as a program that studies the operators does.
        dict(name="setup_acm_7k", kind="setup", solver="acm", cells=20, levels=1, ramp=0.2, r=0.35, n_l=25, k=3, m=2, q=0, steps=0),
        # A new geometry of the high-order cells (N_L = 40, PHS r^5, m = 3), set up and taken a few steps: each
        # cell of a convergence or porosity study pays this once.
        dict(name="setup_acm_r5_86k", kind="setup", solver="acm", cells=25, levels=4, ramp=0.16, r=0.45, n_l=40, k=5, m=3, q=0, steps=8),
        # The lattice Boltzmann set-up of the 120k-node refined cell: 18 interpolation operators per node (N_L = 30).
        dict(name="setup_lbm_120k", kind="setup", solver="lbm", cells=31, levels=3, ramp=0.24, r=0.4, n_l=30, k=3, m=2, q=19, steps=8),
        # The plain FP64 Navier-Stokes solve of the 7k-node cell with its residual checks: small enough that waits
        # and launches count.
        dict(name="acm_solve_fp64_7k", kind="flow", solver="acm", call="solve", prec="fp64", cells=20, levels=1, ramp=0.2, r=0.35,
             n_l=25, k=3, m=2, q=0, steps=200, schedule=0, drag=False),
        # A cell of the warm-start family (40k..150k nodes, N_L = 25) in compensated FP32 from a given start.
        dict(name="acm_solve_fp32c_50k", kind="flow", solver="acm", call="solve", prec="fp32c", cells=25, levels=3, ramp=0.22, r=0.35,
             n_l=25, k=3, m=2, q=0, steps=100, schedule=0, drag=False),
        # The large high-order Navier-Stokes cell in FP32, far larger than the caches.
        dict(name="acm_step_fp32_600k", kind="flow", solver="acm", call="step", prec="fp32", cells=40, levels=5, ramp=0.2, r=0.45,
             n_l=40, k=5, m=3, q=0, steps=32, schedule=0, drag=False),
        # A porosity sweep: cells of different radius, size and stencil in one batched FP32 solve.
        dict(name="batch_fp32_12", kind="batch", n_cells=12, cells_lo=18, cells_hi=26, layout=3, prec="fp32", steps=100, k=3, m=2),
        # The lattice Boltzmann window between two permeability reads on a refined cell of 170k nodes, FP32, schedule as tuned.
        dict(name="lbm_step_fp32_170k", kind="flow", solver="lbm", call="step", prec="fp32", cells=34, levels=3, ramp=0.26, r=0.4,
             n_l=30, k=3, m=2, q=19, steps=100, schedule=10, drag=False),
        # The cross-validation of the paper: D3Q15 in FP64 with permeability and drag, schedule as it comes.
        dict(name="lbm_solve_fp64_17k", kind="flow", solver="lbm", call="solve", prec="fp64", cells=20, levels=2, ramp=0.3, r=0.3,
             n_l=25, k=3, m=2, q=15, steps=100, schedule=0, drag=True),
        # The smallest call: one eager step of a 1.3k-node cell, then permeability and drag.
        dict(name="acm_window_fp64_1k", kind="flow", solver="acm", call="step", prec="fp64", cells=11, levels=1, ramp=0.2, r=0.3,
             n_l=25, k=3, m=2, q=0, steps=1, schedule=0, drag=True),
        # Training of the warm-start network on the nodes of a few solved cells.
        dict(name="mlp_train_16k", kind="train", n=120_000, batch=16384, steps=50),
        # Its prediction at the nodes of a cell of its family.
        dict(name="mlp_predict_60k", kind="predict", n=60_001),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _fit_cells(levels, ramp, r, n):
    """Coarse cells per axis for about n nodes."""
    t = 24
    base = _count(t, levels, ramp, r)
    return max(9, int(round(t * (n / base) ** (1.0 / 3.0))))


def _count(cells, levels, ramp, r):
    return len(_cloud(cells, levels, ramp, r, 0)["xyz"])


def draw(rng):
    kind = rng.choice(["flow"] * 6 + ["setup"] * 3 + ["batch", "train", "predict"])
    if kind == "train":
        return dict(kind=kind, n=int(_log_uniform(rng, 7_000, 120_000)), batch=128 * int(_log_uniform(rng, 4, 128)),
                    steps=rng.randint(10, 50))
    if kind == "predict":
        return dict(kind=kind, n=int(_log_uniform(rng, 1_000, 60_000)))
    if kind == "batch":
        lo = rng.randint(11, 18)
        return dict(kind=kind, n_cells=rng.randint(3, 12), cells_lo=lo, cells_hi=lo + rng.randint(1, 8), layout=rng.randint(0, 1 << 20),
                    prec=rng.choice(["fp32", "fp32", "fp32c", "fp64"]), steps=rng.randint(20, 60), k=3, m=2)
    solver = rng.choice(["acm", "lbm"])
    # the streaming step is unstable on clouds that coarsen faster
    levels, r = rng.randint(1, 5 if solver == "acm" else 2), rng.uniform(0.15, 0.45)
    ramp = rng.uniform(0.15, 0.3)
    high = solver == "acm" and rng.random() < 0.3  # PHS r^5, m = 3
    c = dict(kind=kind, solver=solver, levels=levels, ramp=ramp, r=r, n_l=rng.randint(36, 45) if high else rng.randint(20, 35),
             k=5 if high else 3, m=3 if high else 2, q=rng.choice([15, 19]) if solver == "lbm" else 0)
    if kind == "setup":
        n = _log_uniform(rng, 2_000, 50_000)
        return dict(c, cells=_fit_cells(levels, ramp, r, n), steps=rng.choice([0, 8]) if solver == "acm" and n < 8_000 else 8)
    n = _log_uniform(rng, 1_200, 250_000 if solver == "acm" else 120_000)
    return dict(c, cells=_fit_cells(levels, ramp, r, n), call=rng.choice(["solve", "step"]),
                prec=rng.choice(["fp64", "fp32", "fp32c"] if solver == "acm" else ["fp64", "fp32", "fp32r"]),
                steps=rng.choice([1, 10, 32, 40]) if n > 30_000 else rng.choice([1, 32, 100]),
                schedule=rng.choice([0, 6, 10]) if solver == "lbm" else 0, drag=rng.random() < 0.3)


# ---- one pass ------------------------------------------------------------------------------------

def _pinned(a):
    t = torch.empty(a.shape, dtype=torch.float64, pin_memory=torch.cuda.is_available())
    t.numpy()[...] = a
    return t


def _setup(s, c, cloud):
    """nodes -> stencils -> weights: the calls every program makes first."""
    s.set_case(cloud)
    s.build_stencils(c["n_l"])
    return s.compute_weights(k=c["k"], m=c["m"], solver=rbf.RBF_SOLVER_LBM if c["solver"] == "lbm" else rbf.RBF_SOLVER_ACM,
                             q=c["q"] or 19, dx=0.5 * cloud["h_min"] if c["solver"] == "lbm" else 0.0)


def prepare(case, seed):
    c = case
    rng = np.random.default_rng(seed)
    if c["kind"] == "setup":
        return dict(case=c, cloud=_case_cloud(c, seed))
    if c["kind"] == "train":
        x = rng.random((c["n"], 3))
        rad = rng.uniform(0.15, 0.6, c["n"]).astype(np.float32)
        sdf = rng.uniform(0.0, 0.4, c["n"]).astype(np.float32)
        tgt = (np.sin(2.0 * math.pi * x @ rng.normal(size=(3, 4)).round()) * sdf[:, None] * 3.0).astype(np.float32)
        m = rbf.Mlp()
        m.set_data(x, rad, sdf, tgt)
        return dict(case=c, mlp=m, theta=warmstart.init_params(seed))
    if c["kind"] == "predict":
        x = rng.random((c["n"], 3))
        m = rbf.Mlp()
        m.set_params(warmstart.init_params(seed))
        return dict(case=c, mlp=m, xyz=x, radius=0.35, sdf=rng.uniform(0.0, 0.4, c["n"]).astype(np.float32))
    if c["kind"] == "batch":
        b = rbf.Batch()
        clouds = []
        for j, d in enumerate(_batch_cells(c)):
            clouds.append(_case_cloud(d, seed + 17 * j))
            b.add_cell(clouds[-1], d["n_l"])
        b.build(c["k"], c["m"])
        b.init(precision=PREC[c["prec"]], nu=NU, g=G, v_ref=V_REF)
        return dict(case=c, batch=b, cells=[b.cell(j) for j in range(c["n_cells"])],
                    start=[_pinned(_start_fields(d, seed)) for d in clouds], out=[_pinned(np.zeros((len(d["xyz"]), 4))) for d in clouds])
    cloud = _case_cloud(c, seed)
    s = rbf.Solver()
    if c["solver"] == "lbm" and c["schedule"]:
        s.set_kernel_variant(c["schedule"])
    _setup(s, c, cloud)
    s.init(precision=PREC[c["prec"]], nu=NU, g=G, v_ref=V_REF, tau_plus=TAU, magic=MAGIC)
    start = (_start_fields(cloud, seed) if c["solver"] == "acm"
             else _start_populations(cloud, c["q"], 0.5 * cloud["h_min"], seed))
    return dict(case=c, solver=s, start=_pinned(start), out=_pinned(np.zeros((len(cloud["xyz"]), 4))))


def _fields(s, out, prec):
    f = s.get_fields(out=out.numpy())
    return f if prec == "fp64" else torch.from_numpy(f).float()


def run(state):
    c = state["case"]
    if c["kind"] == "setup":
        s = rbf.Solver()
        rep = _setup(s, c, state["cloud"])
        out = dict(report=rep, stencils=s.get_stencils())
        if c["steps"]:
            s.init(precision=rbf.RBF_FP64, nu=NU, g=G, v_ref=V_REF, tau_plus=TAU, magic=MAGIC)
            s.step(c["steps"])
            out["fields"] = s.get_fields()
        else:
            out["weights"] = [s.get_weights(op) for op in (rbf.RBF_OP_DX, rbf.RBF_OP_DY, rbf.RBF_OP_DZ, rbf.RBF_OP_LAP)]
        s.close()
        return out
    if c["kind"] == "train":
        m = state["mlp"]
        m.set_params(state["theta"])
        hist = m.train(c["steps"], c["batch"], 1e-3, 7)
        return dict(loss=hist, params=m.get_params())
    if c["kind"] == "predict":
        return state["mlp"].predict(state["xyz"], state["radius"], state["sdf"])
    if c["kind"] == "batch":
        for s, f in zip(state["cells"], state["start"]):
            s.set_fields(f.numpy())
        res = state["batch"].solve(c["steps"], 1e-300, check_every=50, m_p=M_P)
        return dict(k=[r["k_over_d2"] for r in res], steps=[r["steps"] for r in res],
                    fields=[_fields(s, o, c["prec"]) for s, o in zip(state["cells"], state["out"])])
    s = state["solver"]
    if c["solver"] == "acm":
        s.set_fields(state["start"].numpy())
    else:
        s.lbm_set_populations(state["start"].numpy())
    if c["call"] == "solve":
        r = s.solve(c["steps"], 1e-300, check_every=50, m_p=M_P)
        out = dict(k=r["k_over_d2"], steps=r["steps"])
    else:
        s.step(c["steps"])
        out = dict(k=s.permeability(M_P)[0])
    if c["drag"]:
        out["force"], out["drag"] = s.drag(M_P)
        if c["prec"] != "fp64":
            out["force"] = out["force"].astype(np.float32)
    out["fields"] = _fields(s, state["out"], c["prec"])
    return out


# ---- what a pass cannot do without -------------------------------------------------------------------

def _acm_bytes(n_l, prec):
    """Per node and step: seven sweeps, each reading its weights and stencil indices once (the predictor 4
    operators, 3 x (pressure, correction) 3 operators each) and its fields once.  A cell that fits on the chip
    can stay below it."""
    return {"fp64": 204 * n_l + 336, "fp32": 116 * n_l + 168, "fp32c": 116 * n_l + 288}[prec]


def work(case):
    c = case
    if c["kind"] == "train":
        return dict(bytes=c["steps"] * (c["batch"] * 48 + 60_000 * 28), flops=c["steps"] * c["batch"] * 356_352)
    if c["kind"] == "predict":
        return dict(bytes=c["n"] * 48 + 240_000, flops=c["n"] * 118_784)
    if c["kind"] == "batch":
        b = f = 0
        for d in _batch_cells(c):
            n = _count(d["cells"], d["levels"], d["ramp"], d["r"])
            b += n * (c["steps"] * _acm_bytes(d["n_l"], c["prec"]) + 64)
            f += n * c["steps"] * 60 * d["n_l"]
        return dict(bytes=b, flops=f)
    n, n_l = _count(c["cells"], c["levels"], c["ramp"], c["r"]), c["n_l"]
    if c["kind"] == "setup":
        ns = n_l + (c["m"] + 1) * (c["m"] + 2) * (c["m"] + 3) // 6
        ops = 4 if c["solver"] == "acm" else c["q"] - 1
        step = c["steps"] * n * (_acm_bytes(n_l, "fp64") if c["solver"] == "acm" else 8 * ((c["q"] - 1) * n_l + 2 * c["q"]) + 4 * n_l)
        # one symmetric factorisation per node, then two triangular solves and a residual per operator
        return dict(bytes=n * (25 + 4 * n_l + 8 * ops * n_l) + step, flops=n * (ns ** 3 / 3 + 6 * ns * ns * ops))
    if c["solver"] == "acm":
        return dict(bytes=n * (c["steps"] * _acm_bytes(n_l, c["prec"]) + 64), flops=n * c["steps"] * 60 * n_l)
    elt, q = (8 if c["prec"] == "fp64" else 4), c["q"]
    per = elt * ((q - 1) * n_l + 2 * q) + 4 * n_l + (4 * q if c["prec"] == "fp32r" else 0)
    return dict(bytes=n * (c["steps"] * per + 8 * q + 32), flops=n * c["steps"] * (2 * (q - 1) * n_l + 300))


# ---- the same results in plain FP64 torch ----------------------------------------------------------------

def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _wrap(d):
    return d - torch.round(d)


def _knn(x, qx, n_l, reach, allow=None):
    """Indices (nq, n_l) of the nearest nodes x of each query, nearest first, over the periodic cell; `reach`
    bounds the n_l-th distance."""
    ids = torch.arange(len(x), device=x.device) if allow is None else torch.nonzero(allow)[:, 0]
    y = x[ids]
    t = max(1, min(8, int(0.5 / reach)))
    tile = torch.clamp((qx * t).long(), 0, t - 1)
    tile = (tile[:, 0] * t + tile[:, 1]) * t + tile[:, 2]
    out = torch.empty((len(qx), n_l), dtype=torch.long, device=x.device)
    for b in torch.unique(tile).tolist():
        mid = (torch.tensor([b // (t * t), b // t % t, b % t], device=x.device, dtype=x.dtype) + 0.5) / t
        near = torch.nonzero((_wrap(y - mid).abs() <= 0.5 / t + reach).all(1))[:, 0]
        rows = torch.nonzero(tile == b)[:, 0]
        for part in torch.split(rows, max(1, 40_000_000 // max(1, len(near)))):
            d2 = sum(_wrap(y[near, a][None, :] - qx[part, a][:, None]) ** 2 for a in range(3))
            v, j = torch.topk(d2, n_l, dim=1, largest=False, sorted=True)
            assert float(v[:, -1].max()) <= reach * reach
            out[part] = ids[near[j]]
    return out


def _monomials(m):
    return [(a, b, d - a - b) for d in range(m + 1) for a in range(d, -1, -1) for b in range(d - a, -1, -1)]


def _weights(x, centre, idx, k, m, ops, node):
    """(n, len(ops), n_l) RBF-FD weights (PHS r^k + monomials up to degree m); an operator is "x", "y", "z",
    "lap" at the centre, or an offset: interpolation there.  Also the scale of each stencil."""
    mono = _monomials(m)
    n, n_l, ns = len(idx), idx.shape[1], idx.shape[1] + len(mono)
    w = torch.empty((n, len(ops), n_l), dtype=x.dtype, device=x.device)
    scale = torch.empty(n, dtype=x.dtype, device=x.device)
    for part in torch.split(torch.arange(n, device=x.device), 4000):
        xi = _wrap(x[idx[part]] - centre[part][:, None, :])
        dl = xi[:, 1 if node else 0].norm(dim=1)
        scale[part] = dl
        xi = xi / dl[:, None, None]
        one = dl.new_ones(len(part))
        M = x.new_zeros((len(part), ns, ns))
        M[:, :n_l, :n_l] = (xi[:, :, None] - xi[:, None, :]).norm(dim=3) ** k
        for j, e in enumerate(mono):
            p = xi[..., 0] ** e[0] * xi[..., 1] ** e[1] * xi[..., 2] ** e[2]
            M[:, :n_l, n_l + j] = p
            M[:, n_l + j, :n_l] = p
        R = x.new_zeros((len(part), ns, len(ops)))
        rho = xi.norm(dim=2)
        for o, op in enumerate(ops):
            if isinstance(op, str) and op == "lap":
                R[:, :n_l, o] = k * (k + 1) * rho ** (k - 2) / dl[:, None] ** 2
                for j, e in enumerate(mono):
                    if sorted(e) == [0, 0, 2]:
                        R[:, n_l + j, o] = 2.0 / dl ** 2
            elif isinstance(op, str):
                a = "xyz".index(op)
                R[:, :n_l, o] = -k * rho ** (k - 2) * xi[..., a] / dl[:, None]
                for j, e in enumerate(mono):
                    if sum(e) == 1 and e[a] == 1:
                        R[:, n_l + j, o] = 1.0 / dl
            else:
                eta = torch.tensor(op, dtype=x.dtype, device=x.device)[None, :] / dl[:, None]
                R[:, :n_l, o] = (eta[:, None, :] - xi).norm(dim=2) ** k
                for j, e in enumerate(mono):
                    R[:, n_l + j, o] = one * eta[:, 0] ** e[0] * eta[:, 1] ** e[1] * eta[:, 2] ** e[2]
        S = torch.linalg.solve(M, R)
        S = S + torch.linalg.solve(M, R - M @ S)
        w[part] = S[:, :n_l].transpose(1, 2)
    return w, scale


class _Exact:
    """One cell in FP64: the stencils, then either solver's steps and the reductions."""

    def __init__(self, cloud, c, h_max):
        t = lambda a: torch.tensor(a, device=_dev())  # noqa: E731
        self.cloud, self.c = cloud, c
        self.x, self.wall, self.nrm = t(cloud["xyz"]), t(cloud["type"]) == 1, t(cloud["normal"])
        self.reach = min(0.45, h_max * (0.9 + 0.9 * c["n_l"] ** (1.0 / 3.0)))
        self.idx = _knn(self.x, self.x, c["n_l"], self.reach)
        self.b = torch.nonzero(self.wall)[:, 0]

    def w(self, ops, idx=None, at=None):
        idx = self.idx if idx is None else idx
        return _weights(self.x, self.x if at is None else self.x[at], idx, self.c["k"], self.c["m"], ops, True)

    def acm(self, f, steps):
        c, fluid = self.c, ~self.wall
        w, scale = self.w(["x", "y", "z", "lap"])
        self.grad = w[:, :3]
        dt, self.h = 0.1 * float(scale.min()) ** 2 / (2.0 * NU), float(scale.min())
        ib = torch.cat([self.b[:, None], _knn(self.x, self.x[self.b], c["n_l"] - 1, self.reach * 1.5, fluid)], 1)
        wn = (self.w(["x", "y", "z"], ib, self.b)[0] * self.nrm[self.b][:, :, None]).sum(1)
        f = torch.tensor(f, device=_dev())
        v, p = f[:, :3].clone(), f[:, 3].clone()
        g = torch.tensor(G, dtype=v.dtype, device=v.device)
        vmax = float(v.norm(dim=1).max())
        for _ in range(steps):
            d = torch.einsum("noj,njc->noc", w, v[self.idx])  # operator o of component c
            vs = v + dt * (NU * d[:, 3] - (v[:, :, None] * d[:, :3]).sum(1) + g)
            vs[self.wall] = 0.0
            v = vs
            for _ in range(3):
                C = 10.0 * max(vmax, V_REF)
                p = torch.where(fluid, p - dt * C * C * (w[:, :3].transpose(1, 2) * v[self.idx]).sum((1, 2)), p)
                p[self.b] = -(wn[:, 1:] * p[ib[:, 1:]]).sum(1) / wn[:, 0]
                v = vs - dt * (w[:, :3] * p[self.idx][:, None, :]).sum(2)
                v[self.wall] = 0.0
                vmax = float(v.norm(dim=1).max())
        self.v, self.p = v, p
        return torch.cat([v, p[:, None]], 1)

    def lbm(self, f, steps):
        c, q = self.c, self.c["q"]
        dx = 0.5 * self.cloud["h_min"]
        e, om = _velocities(q)
        w, scale = self.w([tuple(-dx * e[k]) for k in range(1, q)])
        self.h = float(scale.min())
        dt, gl = _lbm_units(dx)
        et, ot, gt = (torch.tensor(a, device=_dev()) for a in (e, om, gl))
        tp, tm = TAU, 0.5 + MAGIC / (TAU - 0.5)
        opp = torch.tensor([0] + [k + 1 if k % 2 else k - 1 for k in range(1, q)], device=_dev())
        un = ((self.nrm @ et.T) > 0) & self.wall[:, None]

        def collide(h):  # h: populations less their weights, (n, q)
            drho = h.sum(1)
            rho = 1.0 + drho
            v = (h @ et) / rho[:, None]
            eu, vv = v @ et.T, (v * v).sum(1)
            eq = ot * (drho[:, None] + rho[:, None] * (3.0 * eu + 4.5 * eu * eu - 1.5 * vv[:, None]))
            dh = h - eq
            return h - 0.5 * (dh + dh[:, opp]) / tp - 0.5 * (dh - dh[:, opp]) / tm + ot * 3.0 * rho[:, None] * (et @ gt)

        if f is None:
            h = collide(torch.zeros((len(self.x), q), dtype=self.x.dtype, device=_dev()))
        else:
            h = torch.tensor(f, device=_dev()).T - ot
        for _ in range(steps):
            s = torch.empty_like(h)
            s[:, 0] = h[:, 0]
            for k in range(1, q):
                s[:, k] = (w[:, k - 1] * h[:, k][self.idx]).sum(1)
            h = collide(torch.where(un, s[:, opp], s))
        drho = h.sum(1)
        vel = dx / dt
        self.v = ((h @ et) / (1.0 + drho)[:, None] - gt) * vel
        self.p = (drho - drho.mean()) / (1.0 + drho.mean()) / 3.0 * vel * vel
        return torch.cat([self.v, self.p[:, None]], 1)

    def flux(self):
        a = (torch.arange(M_P, device=_dev(), dtype=self.x.dtype) + 0.5) / M_P
        pts = torch.stack(torch.meshgrid(0.2 * torch.arange(5, device=_dev(), dtype=self.x.dtype), a, a, indexing="ij"), -1).reshape(-1, 3)
        pts = pts[_wrap(pts - 0.5).norm(dim=1) >= self.cloud["radius"]]
        idx = _knn(self.x, pts, self.c["n_l"], self.reach * 1.5)
        w, _ = _weights(self.x, pts, idx, self.c["k"], self.c["m"], [(0.0, 0.0, 0.0)], False)
        return float((w[:, 0] * self.v[idx, 0]).sum()) / (5.0 * M_P * M_P)

    def drag(self, flux):
        r, ib, n = self.cloud["radius"], self.idx[self.b], self.nrm[self.b]
        d = torch.einsum("noj,njc->nco", self.w(["x", "y", "z"], ib, self.b)[0], self.v[ib])  # d v_c / d x_o
        p = self.p[self.b]
        s = -p[:, None] * n + NU * ((d + d.transpose(1, 2)) * n[:, None, :]).sum(2)
        F = 4.0 * math.pi * r * r / len(n) * (s.sum(0) + p.mean() * n.sum(0))
        return F.cpu().numpy(), float(F[0]) / (6.0 * math.pi * r * (1.0 - 4.0 / 3.0 * math.pi * r ** 3) * flux * NU)


def exact(case, seed):
    c = case
    if c["kind"] == "train":  # tens of optimiser steps on 16-bit operands: no value to hold a run to
        return None
    if c["kind"] == "predict":
        s = prepare(c, seed)
        th = warmstart.init_params(seed).astype(np.float64)
        waves = np.array([(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1), (1, 1, 1),
                          (1, 1, -1), (1, -1, 1), (1, -1, -1), (2, 0, 0), (0, 2, 0), (0, 0, 2)], np.float64)
        ph = 2.0 * math.pi * s["xyz"] @ waves.T
        h = np.zeros((c["n"], 64))
        h[:, 0:32:2], h[:, 1:32:2], h[:, 32], h[:, 33] = np.sin(ph), np.cos(ph), s["radius"], s["sdf"]
        o = 0
        for j, (fi, fo) in enumerate(warmstart.LAYERS):
            h = h @ th[o:o + fo * fi].reshape(fo, fi).T + th[o + fo * fi:o + fo * fi + fo]
            o += fo * fi + fo
            if j < 4:
                h = 0.5 * h * (1.0 + np.tanh(math.sqrt(2.0 / math.pi) * (h + 0.044715 * h ** 3)))
        return h[:, :4]
    if c["kind"] == "batch":
        out = dict(k=[], steps=None, fields=[])
        for j, d in enumerate(_batch_cells(c)):
            cloud = _case_cloud(d, seed + 17 * j)
            x = _Exact(cloud, dict(d, k=c["k"], m=c["m"]), 1.0 / d["cells"])
            out["fields"].append(x.acm(_start_fields(cloud, seed), c["steps"]))
            out["k"].append(x.flux() * NU)
        return out
    cloud = _case_cloud(c, seed)
    x = _Exact(cloud, c, 1.0 / c["cells"])
    if c["kind"] == "setup":
        if not c["steps"]:
            w, scale = x.w(["x", "y", "z", "lap"])
            return dict(report=dict(n_systems=None, n_singular=None, h_min=float(scale.min())), stencils=None,
                        weights=[w[:, j].contiguous() for j in range(4)])
        f = x.acm(np.zeros((len(cloud["xyz"]), 4)), c["steps"]) if c["solver"] == "acm" else x.lbm(None, c["steps"])
        return dict(report=dict(n_systems=None, n_singular=None, h_min=x.h), stencils=None, fields=f)
    if c["solver"] == "acm":
        f = x.acm(_start_fields(cloud, seed), c["steps"])
    else:
        f = x.lbm(_start_populations(cloud, c["q"], 0.5 * cloud["h_min"], seed), c["steps"])
    flux = x.flux()
    out = dict(k=flux * NU, steps=None, fields=f)
    if c["drag"]:
        out["force"], out["drag"] = x.drag(flux)
    return out
