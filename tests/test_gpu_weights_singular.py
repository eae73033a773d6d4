"""Exactly singular stencil systems are found, all of them: a cloud with coincident nodes (two equal
rows in every stencil that holds both), and lattice clouds on which the stencils' polynomial
columns are linearly dependent (their rank evaluated in integers), through the FP32 inverse
(r^3, r^5) and the FP64 factors alone (r^7, r^9).  Counts, so no tolerance.
"""
import ctypes

import numpy as np
import pytest

import oracle
from gpu_common import gpu_or_skip

pytestmark = pytest.mark.gpu


def _count(rbf, xyz, n_l, k, m):
    s = rbf.Solver(0)
    s.set_nodes(xyz, np.zeros(len(xyz), np.uint8))
    s.build_stencils(n_l)
    rep = rbf.rbf_weight_report()
    rc = s._L.rbf_compute_weights(s._h, k, m, rbf.RBF_SOLVER_ACM, 0, 0.0, ctypes.byref(rep))
    idx = s.get_stencils()
    s.close()
    assert rc == (rbf.RBF_ESINGULAR if rep.n_singular else rbf.RBF_OK)
    return rep.n_singular, idx


def _grid(n):
    return np.stack(np.meshgrid(*[np.arange(n)] * 3, indexing="ij"), -1).reshape(-1, 3)


@pytest.mark.parametrize("n_l,k,m", [(25, 3, 2), (40, 5, 3), (64, 5, 4), (64, 3, 4), (35, 7, 3), (40, 9, 3)])
def test_coincident_nodes(n_l, k, m):
    rbf = gpu_or_skip()
    rng = np.random.default_rng(0)
    x = (_grid(9) + 0.5 + rng.uniform(-0.2, 0.2, (729, 3))) / 9
    twin = rng.choice(len(x), 12, replace=False)
    n_sing, idx = _count(rbf, np.vstack([x, x[twin]]), n_l, k, m)
    both = np.zeros(len(idx), bool)
    for j, i in enumerate(twin):
        both |= (idx == i).any(1) & (idx == len(x) + j).any(1)
    assert both.sum() > 200 and n_sing == both.sum()


def _rank(rows, p=(1 << 61) - 1):
    """Rank of an integer matrix modulo the prime p (its entries are far below p)."""
    a, rank = [[int(v) % p for v in r] for r in rows], 0
    for c in range(len(a[0])):
        q = next((r for r in range(rank, len(a)) if a[r][c]), None)
        if q is None:
            continue
        a[rank], a[q] = a[q], a[rank]
        inv = pow(a[rank][c], p - 2, p)
        for r in range(rank + 1, len(a)):
            f = a[r][c] * inv % p
            if f:
                a[r] = [(u - f * v) % p for u, v in zip(a[r], a[rank])]
        rank += 1
    return rank


@pytest.mark.parametrize("k", [3, 5, 7, 9])
@pytest.mark.parametrize("n_l,m,want", [(30, 3, 384), (26, 3, 512), (14, 2, 64), (33, 3, 0)])
def test_dependent_polynomials(n_l, m, want, k):
    rbf = gpu_or_skip()
    g = _grid(8)
    x = (g + 0.5) / 8  # exact in FP64
    n_sing, idx = _count(rbf, x, n_l, k, m)
    assert np.array_equal(idx, oracle.knn(x, x, n_l))
    mono = [(a, b, d - a - b) for d in range(m + 1) for a in range(d, -1, -1) for b in range(d - a, -1, -1)]
    known, deficient = {}, 0
    for i in range(512):
        o = (g[idx[i]] - g[i] + 4) % 8 - 4
        key = o.tobytes()
        if key not in known:
            known[key] = _rank([[p[0] ** e[0] * p[1] ** e[1] * p[2] ** e[2] for e in mono] for p in o.tolist()]) < len(mono)
        deficient += known[key]
    assert deficient == want  # the count in integers
    assert n_sing == want
