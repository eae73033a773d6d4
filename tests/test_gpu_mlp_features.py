"""The input features of a prediction, bit for bit, and its outputs in the mean.

Features: a network that carries four chosen inputs through its layers unchanged.  Each input f is
split into 2^20 f and -2^20 f, whose GELUs are 2^20 max(f, 0) and 2^20 max(-f, 0) once
|2^20 f| >= 16 (there the GELU is x or 0 to the last FP32 bit); the hidden layers copy, the
output layer takes the difference times 2^-20.  All factors are powers of two and every sum has one
nonzero term, so the output is the BF16 input itself, which has to equal the FP64 feature
rounded to BF16: random points, phases that are multiples of 1/8, and phases at BF16 rounding
boundaries +- 1e-11 .. 3e-7 (the reference is good to 1e-15).

Outputs of a random network against the FP64 layers with BF16 rounding points: a different
accumulation order moves a rounding now and then, so the largest error grows with the number of
points; evaluated on the CPU (FP32 sums in three orders, the same points) the largest of 60,001 is
4.2e-3 of the largest output and the root mean square 5.7e-5, while one input in a hundred
off by one BF16 ulp gives 5.3e-4: twice the first, and 2e-4 in the mean.
"""
import numpy as np
import pytest

from gpu_common import bf16_forward, gpu_or_skip
from oracle import mlp as om

pytestmark = pytest.mark.gpu


def _selector(columns):
    """Packed parameters of the network whose outputs are the given input columns."""
    layers = []
    for li, (fo, fi) in enumerate(om.param_sizes()):
        w = np.zeros((fo, fi))
        for j, c in enumerate(columns):
            if li == 0:
                w[2 * j, c], w[2 * j + 1, c] = 2.0 ** 20, -2.0 ** 20
            elif li < 4:
                w[2 * j, 2 * j] = w[2 * j + 1, 2 * j + 1] = 1.0
            else:
                w[j, 2 * j], w[j, 2 * j + 1] = 2.0 ** -20, -2.0 ** -20
        layers += [w.ravel(), np.zeros(fo)]
    return np.concatenate(layers).astype(np.float32)


def _sincospi(t):
    """sin and cos of pi t, exact where they are 0 or +-1."""
    t = t - 2.0 * np.rint(t / 2.0)  # [-1, 1]
    a = np.abs(t)
    b = np.where(a > 0.5, 1.0 - a, a)  # [0, 1/2]
    low = b <= 0.25
    s = np.where(low, np.sin(np.pi * b), np.cos(np.pi * (0.5 - b)))
    c = np.where(low, np.cos(np.pi * b), np.sin(np.pi * (0.5 - b)))
    return np.copysign(s, t), np.where(a > 0.5, -c, c)


def _points():
    rng = np.random.default_rng(11)
    out = [rng.random((6000, 3)), rng.integers(-16, 17, (3000, 3)) / 8.0, 4.0 * rng.random((3000, 3)) - 2.0]
    m = (rng.integers(128, 256, 6000) * 2 + 1) * 2.0 ** -(9 + rng.integers(0, 7, 6000))  # between two BF16 values
    x = np.arcsin(m) / (2.0 * np.pi) + rng.choice([1e-11, 1e-9, 1e-8, 1e-7, 3e-7], len(m)) * rng.choice([-1.0, 1.0], len(m))
    p = np.zeros((len(m), 3))
    p[np.arange(len(m)), rng.integers(0, 3, len(m))] = np.where(rng.random(len(m)) < 0.5, x, x + 0.25)  # a sine or a cosine
    return np.concatenate(out + [p])


def _bf16(v):
    """FP64 to BF16 in one rounding (the oracle's bf16_round goes through FP32 first)."""
    m, e = np.frexp(v)
    return np.ldexp(np.rint(m * 256.0) / 256.0, e)


def test_feature_bits():
    rbf = gpu_or_skip()
    xyz = _points()
    rng = np.random.default_rng(12)
    n = len(xyz)
    rad, sdf = rng.uniform(0.15, 0.6, n).astype(np.float32), rng.uniform(0.0, 0.4, n).astype(np.float32)
    want = np.zeros((n, 36))
    w = om.WAVES
    ph = (w[:, 0] * xyz[:, :1] + w[:, 1] * xyz[:, 1:2]) + w[:, 2] * xyz[:, 2:]
    want[:, 0:32:2], want[:, 1:32:2] = _sincospi(2.0 * ph)
    want[:, 32], want[:, 33] = rad, sdf
    m = rbf.Mlp(0)
    near = 0
    for c0 in range(0, 36, 4):
        m.set_params(_selector(range(c0, c0 + 4)))
        got = m.predict(xyz, rad, sdf).astype(np.float64)
        f = want[:, c0:c0 + 4]
        b = _bf16(f)
        # where the GELU is exact, and the reference's own error cannot move the rounding
        exact = ((f == 0.0) | (np.abs(f) >= 2.0 ** -16)) & (np.abs(_bf16(f * (1 + 4e-15)) - _bf16(f * (1 - 4e-15))) == 0.0)
        near += int((np.abs(_bf16(f * (1 + 1e-6)) - _bf16(f * (1 - 1e-6))) != 0.0).sum())
        assert exact.mean() > 0.99
        assert np.array_equal(got[exact], b[exact]), (c0, np.abs(got - b)[exact].max())
        assert np.abs(got - b).max() <= 2.0 ** -16
    assert near > 3000  # values at a rounding boundary were among them
    m.close()


@pytest.mark.parametrize("n", [5000, 60001])
def test_outputs_in_the_mean(n):
    rbf = gpu_or_skip()
    rng = np.random.default_rng(n)
    xyz = rng.random((n, 3))
    xyz[: n // 8] = np.round(xyz[: n // 8] * 8) / 8
    rad, sdf = rng.uniform(0.15, 0.6, n).astype(np.float32), rng.uniform(0.0, 0.4, n).astype(np.float32)
    theta = om.init_params(3).astype(np.float32)
    m = rbf.Mlp(0)
    m.set_params(theta)
    want = bf16_forward(theta.astype(np.float64), om.bf16_round(om.features(xyz, rad, sdf)))
    e = np.abs(m.predict(xyz, rad, sdf) - want) / np.abs(want).max()
    assert e.max() <= 8.4e-3 and np.sqrt((e ** 2).mean()) <= 2e-4
    m.close()
