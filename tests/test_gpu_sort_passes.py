"""Preparation's sort at the sizes where its passes over the data take one, two
or three levels: no point is lost (the histograms equal the oracle's) and the
order is spatial (pruning leaves out most pairs of a full sky at small angles)."""
import os

import numpy as np
import pytest

import oracle
from paper_1204_6630_gb300 import build, synth

pytestmark = pytest.mark.gpu
THREADS = os.cpu_count() or 4


@pytest.mark.parametrize("n", [2047, 2049, 4097, 8193, 16385, 33000, 66001])
def test_sorted(n):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    from paper_1204_6630_gb300 import tpcf as T
    T.load()
    d = synth.randoms(n, synth.Footprint("sphere"), seed=n)
    edges = synth.log_edges(0.05, 1.0, 5)
    with T.Context(flags=T.TPCF_F_PRUNE) as ctx:
        got, st = ctx.count_auto(ctx.catalog(d), ctx.bins(edges), stats=True)
    np.testing.assert_array_equal(got, oracle.count_auto(d, edges, THREADS))
    # a group of 128 sorted points spans about 2 sqrt(512 / n) radians and meets few of the others
    if n > 8000:
        assert st["pruned_pairs"] > 0.5 * st["pairs"]
