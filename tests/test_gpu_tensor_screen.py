"""The tensor-core counting kernel (the default for angular catalogs) at the
edges of its tiles: 32 x 32 blocks, groups of 128 and items of 512 i-points,
tiles of 128 and chunks of up to 4096 j-points, with and without pruning and
with a counted overflow row; every histogram equals the oracle's integer for
integer."""
import os

import numpy as np
import pytest

import oracle
from paper_1204_6630_gb300 import build, synth

pytestmark = pytest.mark.gpu
THREADS = os.cpu_count() or 4


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
        cd, cr, b = ctx.catalog(d), ctx.catalog(r), ctx.bins(edges)
        got, st = ctx.count_all(cd, cr, b, stats=True)
        dr = ctx.count_cross(cd, cr, b)
    want = (oracle.count_auto(d, edges, THREADS), oracle.count_cross(d, r, edges, THREADS),
            oracle.count_auto(r, edges, THREADS))
    for g, o in zip(got, want):
        np.testing.assert_array_equal(g, o)
    np.testing.assert_array_equal(dr, want[1])
    assert st["device_error"] == 0
    assert st["pairs"] == sum(int(o.sum()) for o in want)


SIZES = [(1, 33), (31, 32), (128, 127), (129, 511), (513, 512), (640, 4097), (1025, 129)]


@pytest.mark.parametrize("mode", ["plain", "prune", "check"])
@pytest.mark.parametrize("nd,nr", SIZES)
def test_tile_edges(T, nd, nr, mode):
    flags = {"plain": 0, "prune": T.TPCF_F_PRUNE, "check": T.TPCF_F_CHECK_OVERFLOW}[mode]
    d = synth.clustered(nd, 8, 0.5, seed=nd)
    r = synth.randoms(nr, seed=nr)
    _check(T, d, r, synth.log_edges(0.05, 6.0, 17), flags=flags)


@pytest.mark.parametrize("hi", [0.02, 1.0, 89.9999, 90.0, 179.0])
def test_range_ends(T, hi):
    """The rejection threshold from ranges far below its guard to ranges that reject nothing
    (past 90 degrees zero-vector padding looks in range)."""
    d = synth.clustered(700, 8, 0.01, synth.Footprint("sphere"), seed=3)
    r = np.concatenate([synth.randoms(600, synth.Footprint("sphere"), seed=4), -d[:50], d[:50]])
    _check(T, d, r, synth.linear_edges(0.0, hi, 7))


@pytest.mark.parametrize("flags", [0, 0x10, 0x20])
def test_chunks_of_several_tiles(T, flags):
    """Large enough for chunks of more than one tile and, with pruning, batched draws; with a
    counted overflow row most tiles are whole ones that hold nothing in range."""
    fp = synth.Footprint("sphere")
    d = synth.clustered(30011, 64, 0.5, fp, seed=8)
    r = synth.randoms(41001, fp, seed=9)
    _check(T, d, r, synth.log_edges(0.05, 3.0, 21), flags=flags)


def test_values_at_the_threshold(T):
    """Pairs placed within a few units of the last edge, on both sides, are classified exactly."""
    rng = np.random.default_rng(5)
    tb = np.radians(2.0)
    a = synth.randoms(256, synth.Footprint("sphere"), seed=6)
    t = rng.normal(size=a.shape)
    t -= (t * a).sum(1)[:, None] * a
    t /= np.linalg.norm(t, axis=1)[:, None]
    ang = tb + np.concatenate([np.linspace(-4e-6, 4e-6, 192), np.zeros(64)])
    b = np.cos(ang)[:, None] * a + np.sin(ang)[:, None] * t
    b /= np.linalg.norm(b, axis=1)[:, None]
    _check(T, a, b, np.linspace(0.0, tb, 9))


@pytest.mark.parametrize("nedges", [110, 111, 121, 122, 132, 133])
def test_ring_depths(T, nedges):
    """Histograms take shared memory from the ring of tiles: eight stages up to 110 edges, six up
    to 121, four up to 132, beyond that the FP32 kernel; many more tiles than stages in each."""
    d = synth.clustered(2003, 8, 0.5, seed=nedges)
    r = synth.randoms(9001, seed=nedges + 1)
    _check(T, d, r, synth.linear_edges(0.0, 20.0, nedges - 1))


def test_a_short_wait_limit_outlasts_slow_tiles(T):
    """Points a few arc seconds apart: nearly every pair goes to binary64 and a tile takes
    milliseconds.  The limit of the device's waits counts time without progress, so one far
    shorter than a tile still holds."""
    d = synth.randoms(20000, synth.Footprint("sphere"), seed=5)
    c = np.array([0.48, 0.6, 0.64])
    d = c + 1e-5 * d
    d /= np.linalg.norm(d, axis=1)[:, None]
    edges = np.linspace(0.0, 2e-5, 100)
    with T.Context(wait_timeout_us=300) as ctx:
        got = ctx.count_auto(ctx.catalog(d), ctx.bins(edges))
    np.testing.assert_array_equal(got, oracle.count_auto(d, edges, THREADS))
