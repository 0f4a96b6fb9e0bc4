"""The all-binary64 mode where its comparisons and launch shapes can go wrong:
dots of both signs and exactly zero against thresholds of both signs, 128, 256
and 512 threads, chunks of one tile and more; every histogram equals the
oracle's integer for integer."""
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


@pytest.mark.parametrize("lo,hi", [(0.0, 1.0), (0.5, 90.0), (90.0, 90.5), (89.0, 179.0), (0.0, 180.0)])
@pytest.mark.parametrize("n", [200, 7001, 12000])
def test_plain(T, n, lo, hi):
    fp = synth.Footprint("sphere")
    axes = np.concatenate([np.eye(3), -np.eye(3), [[0.6, 0.8, 0.0], [-0.8, 0.6, 0.0]]])  # dots of exactly 0 and -0
    d = np.concatenate([synth.clustered(n, 16, 0.5, fp, seed=n), axes])
    r = np.concatenate([synth.randoms(n // 2 + 3, fp, seed=n + 1), axes])
    edges = np.radians(np.linspace(lo, hi, 10)).clip(max=np.pi)
    with T.Context(precision=1) as ctx:
        got, st = ctx.count_all(ctx.catalog(d), ctx.catalog(r), ctx.bins(edges), stats=True)
    want = (oracle.count_auto(d, edges, THREADS), oracle.count_cross(d, r, edges, THREADS),
            oracle.count_auto(r, edges, THREADS))
    for g, o in zip(got, want):
        np.testing.assert_array_equal(g, o)
    assert st["device_error"] == 0
