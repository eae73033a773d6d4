"""Prediction over its range of point counts (below, at and past a 128-row tile, one and two tile
groups per block) against the FP64 network with the kernels' BF16 rounding points.

Tolerance: as for the other forward test, 2e-2 of the largest output: BF16 activations (2^-9 each)
through four hidden layers, where a different accumulation order can move a rounding.
"""
import numpy as np
import pytest

from gpu_common import bf16_forward, gpu_or_skip, rel_inf
from oracle import mlp as om

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 127, 128, 129, 5000, 152 * 128, 152 * 128 + 1, 60001])
def test_predict_counts(n):
    rbf = gpu_or_skip()
    rng = np.random.default_rng(n)
    xyz = rng.random((n, 3))
    xyz[: n // 8] = np.round(xyz[: n // 8] * 8) / 8  # phases whose sine or cosine is exactly 0 or +-1
    rad, sdf = rng.uniform(0.15, 0.6, n).astype(np.float32), rng.uniform(0.0, 0.4, n).astype(np.float32)
    theta = om.init_params(3).astype(np.float32)
    m = rbf.Mlp(0)
    m.set_params(theta)
    for _ in range(2):  # the second call reuses the workspace
        got = m.predict(xyz, rad, sdf)
    want = bf16_forward(theta.astype(np.float64), om.bf16_round(om.features(xyz, rad, sdf)))
    assert got.shape == (n, 4) and rel_inf(got, want) <= 2e-2
    # a point's output does not depend on the others of the call
    k = min(n, 130)
    assert np.array_equal(m.predict(xyz[:k], rad[:k], sdf[:k]), got[:k])
    m.close()
