"""The values by which the tensor-core kernel rejects, read out of its product and
compared with binary64: within the bounds that its thresholds rest on (44u for
angles, 49u max(s, 1/s) for 3-D points, of which all but 12u and 12 + 5s u is
the unit's accumulation), and their maxima of 32 are those of the values."""
import math

import numpy as np
import pytest

from paper_1204_6630_gb300 import build, synth

pytestmark = pytest.mark.gpu
U = 2.0 ** -24
BLOCKS = 6  # of 128 points


@pytest.fixture(scope="module")
def T():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    from paper_1204_6630_gb300 import tpcf
    tpcf.load()
    return tpcf


def _values(T, ctx, a, b):
    for i in range(BLOCKS):
        for j in range(BLOCKS):
            v, m = T.tpcf_debug_screen_values(ctx.handle, a.handle, b.handle, i, j)
            np.testing.assert_array_equal(m, v.reshape(128, 4, 32).max(2))
            yield slice(128 * i, 128 * i + 128), slice(128 * j, 128 * j + 128), v.astype(np.float64)


def _sky(name, seed):
    n, rng = 128 * BLOCKS, np.random.default_rng(seed)
    if name == "sphere":
        return synth.randoms(n, synth.Footprint("sphere"), seed)
    if name == "octant":
        return synth.clustered(n, 16, 0.2, synth.Footprint("octant"), seed)
    p = np.array([0.48, 0.6, 0.64]) if name == "cap" else np.eye(3)[rng.integers(0, 3, n)]  # a few arc seconds; the axes
    p = p + rng.normal(0.0, 1e-5, (n, 3))
    return p / np.linalg.norm(p, axis=1, keepdims=True)


@pytest.mark.parametrize("name", ["sphere", "octant", "cap", "axes"])
def test_angular_values(T, name):
    a, b = _sky(name, 1), _sky(name, 2)
    b[::3] *= -1.0 if name == "sphere" else 1.0
    worst = 0.0
    with T.Context(flags=T.TPCF_F_NO_SORT) as ctx:
        for i, j, v in _values(T, ctx, ctx.catalog(a), ctx.catalog(b)):
            worst = max(worst, np.abs(v - a[i] @ b[j].T).max() / U)
    print(f"{name}: largest error {worst:.2f} u")
    assert worst <= 44.0


def _exponent(p):
    return (math.floor(math.log2((p * p).sum(1).max())) + 2) >> 1


@pytest.mark.parametrize("scale", [1.0, 1e6])
@pytest.mark.parametrize("ratio", [-10, -3, 0, 3, 10])
def test_3d_values(T, ratio, scale):
    rng = np.random.default_rng(ratio + 30)
    a = scale * rng.uniform(-0.5, 0.5, (128 * BLOCKS, 3))
    b = scale * 2.0 ** ratio * rng.uniform(-0.5, 0.5, (128 * BLOCKS, 3))
    ka, kb = _exponent(a), _exponent(b)
    assert abs(kb - ka) <= 10
    s, worst = 2.0 ** (kb - ka), 0.0
    with T.Context(flags=T.TPCF_F_NO_SORT) as ctx:
        for i, j, v in _values(T, ctx, ctx.catalog3d(a), ctx.catalog3d(b)):
            want = (a[i] @ b[j].T - 0.5 * (b[j] * b[j]).sum(1)) * 2.0 ** -(ka + kb)
            worst = max(worst, np.abs(v - want).max() / U)
    print(f"ratio {ratio}: largest error {worst:.2f} u, {worst / max(s, 1 / s):.2f} u max(s, 1/s)")
    assert worst <= 49.0 * max(s, 1.0 / s)
