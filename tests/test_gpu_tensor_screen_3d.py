"""The tensor-core screen of 3-D counts: its error bound without the
accumulation (on the CPU, a binary16 split as the preparation writes it), and
on the GPU every histogram against the oracle at the tiles' edges, over scales,
catalogs of different scales and distances from the origin on both sides of
the rule that chooses it."""
import os

import numpy as np
import pytest

import oracle
from paper_1204_6630_gb300 import build, synth

THREADS = os.cpu_count() or 4
U = 2.0 ** -24


def _split(v):
    hi = v.astype(np.float16)
    lo = (v - hi.astype(np.float32)).astype(np.float16)
    return hi.astype(np.float64), lo.astype(np.float64)


@pytest.mark.parametrize("ratio", [-10, -3, 0, 1, 10])
def test_value_error(ratio):
    """|value - exact| <= (2 + 9.8 + 5 s) u for points of norm <= 1 (no accumulation error)."""
    rng = np.random.default_rng(ratio + 20)
    s = 2.0 ** ratio
    a, b = rng.normal(size=(2, 4000, 3))
    a *= (rng.random((4000, 1)) ** 0.3) / np.linalg.norm(a, axis=1, keepdims=True)
    b *= (rng.random((4000, 1)) ** 0.3) / np.linalg.norm(b, axis=1, keepdims=True)
    exact = (a * b).sum(1) - s * (b * b).sum(1) / 2
    a32, b32 = a.astype(np.float32), b.astype(np.float32)
    (ah, al), (bh, bl) = _split(a32), _split(b32)
    nh, nl = _split(np.float32(-0.5) * (b32 * b32).sum(1))
    value = ((ah + al) * (bh + bl)).sum(1) + s * (nh + nl)
    assert np.abs(value - exact).max() <= (2 + 9.8 + 5 * s) * U


@pytest.fixture(scope="module")
def T():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    from paper_1204_6630_gb300 import tpcf
    tpcf.load()
    return tpcf


def _check(T, d, r, edges, **kw):
    with T.Context(**kw) as ctx:
        got, st = ctx.count_all(ctx.catalog3d(d), ctx.catalog3d(r), ctx.bins3d(edges), stats=True)
    want = (oracle.count_auto(d, edges, THREADS, euclid=True), oracle.count_cross(d, r, edges, THREADS, euclid=True),
            oracle.count_auto(r, edges, THREADS, euclid=True))
    for g, o in zip(got, want):
        np.testing.assert_array_equal(g, o)
    assert st["device_error"] == 0


@pytest.mark.gpu
@pytest.mark.parametrize("mode", ["plain", "prune", "check"])
@pytest.mark.parametrize("nd,nr", [(1, 33), (128, 127), (513, 512), (640, 4097)])
def test_tile_edges(T, nd, nr, mode):
    flags = {"plain": 0, "prune": T.TPCF_F_PRUNE, "check": T.TPCF_F_CHECK_OVERFLOW}[mode]
    d = synth.box_clustered(nd, 8, 0.5, 100.0, nd)
    r = synth.box_points(nr, 100.0, nr)
    _check(T, d, r, synth.log_edges_r(0.3, 12.0, 17), flags=flags)


@pytest.mark.gpu
@pytest.mark.parametrize("scale", [1e-10, 1.0, 1e12])
@pytest.mark.parametrize("ratio", [0.0005, 0.1, 30.0, 3000.0])
@pytest.mark.parametrize("offset", [0.0, 20.0, 2000.0])
def test_scales(T, scale, ratio, offset):
    """The second catalog's extent is `ratio` times the first's; both lie `offset` extents off the origin."""
    d = scale * (synth.box_clustered(900, 8, 0.02, 1.0, 5) + offset)
    r = scale * (ratio * synth.box_points(1100, 1.0, 6) + offset)
    _check(T, d, r, scale * synth.log_edges_r(0.005, 0.3, 9))


@pytest.mark.gpu
@pytest.mark.parametrize("hi", [1e-7, 0.004, 0.5, 3.0])
def test_range_ends(T, hi):
    """Ranges below the screen's band, around it, and past every pair."""
    d = synth.box_clustered(700, 8, 0.01, 1.0, 3) - 0.5
    r = np.concatenate([synth.box_points(600, 1.0, 4) - 0.5, d[:50], d[:50] + 1e-8])
    _check(T, d, r, np.linspace(0.0, hi, 8))


@pytest.mark.gpu
def test_autotuned_shapes(T):
    """A shape tuned on points near the origin is not used for points the screen refuses."""
    d, r = synth.box_clustered(3000, 8, 0.02, 1.0, 5), synth.box_points(3100, 1.0, 6)
    edges = synth.log_edges_r(0.005, 0.3, 9)
    with T.Context(flags=T.TPCF_F_AUTOTUNE) as ctx:
        for offset in (0.0, 5e5, 0.0):
            a, b = d + offset, r + offset
            got = ctx.count_all(ctx.catalog3d(a), ctx.catalog3d(b), ctx.bins3d(edges))
            want = (oracle.count_auto(a, edges, THREADS, euclid=True),
                    oracle.count_cross(a, b, edges, THREADS, euclid=True),
                    oracle.count_auto(b, edges, THREADS, euclid=True))
            for g, o in zip(got, want):
                np.testing.assert_array_equal(g, o)
