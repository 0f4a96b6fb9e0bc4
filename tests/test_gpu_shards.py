"""The counting kernel on shards of the pair space (tpcf_config.shard_index /
shard_count, one process per GPU in production; here every shard runs in
turn on one GPU): the shards' histograms sum to the unsplit ones, which equal
the oracle's; with more items than blocks, so the dynamic item draws of every
shard's launch are exercised."""
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


def _count(T, d, r, edges, **kw):
    with T.Context(**kw) as ctx:
        (dd, dr, rr), st = ctx.count_all(ctx.catalog(d), ctx.catalog(r), ctx.bins(edges), stats=True)
    assert st["device_error"] == 0
    return np.stack([dd, dr, rr]), st["pairs"]


@pytest.mark.parametrize("world", [2, 3, 5])
def test_shards_sum_to_the_unsplit_histograms(T, world):
    d = synth.clustered(60000, 256, 0.3, seed=21)
    r = synth.randoms(90000, seed=22)
    edges = synth.log_edges(0.02, 6.0, 30)
    full, pairs = _count(T, d, r, edges, threads=128, ipt=8)
    parts = [_count(T, d, r, edges, threads=128, ipt=8, shard_index=s, shard_count=world) for s in range(world)]
    np.testing.assert_array_equal(np.sum([p[0] for p in parts], axis=0, dtype=np.uint64), full)
    assert sum(p[1] for p in parts) == pairs


def test_shards_against_the_oracle(T):
    w = synth.octant_small(seed=5, n=6000)
    want = np.stack([oracle.count_auto(w.data, w.edges, THREADS), oracle.count_cross(w.data, w.rand, w.edges, THREADS),
                     oracle.count_auto(w.rand, w.edges, THREADS)])
    parts = [_count(T, w.data, w.rand, w.edges, threads=128, ipt=8, shard_index=s, shard_count=3)[0] for s in range(3)]
    np.testing.assert_array_equal(np.sum(parts, axis=0, dtype=np.uint64), want)


def test_shards_of_autotuned_contexts_cut_the_work_alike(T):
    """A context that tuned a smaller problem of the same class first (whose items are
    smaller) still takes the same items as the other shards' contexts."""
    edges = synth.log_edges(0.02, 6.0, 30)
    small, x = synth.randoms(17000, seed=23), synth.clustered(20000, 64, 0.3, seed=24)
    parts = []
    for s in range(2):
        with T.Context(flags=T.TPCF_F_AUTOTUNE, shard_index=s, shard_count=2) as ctx:
            b = ctx.bins(edges)
            if s == 0:
                ctx.count_auto(ctx.catalog(small), b)
            parts.append(ctx.count_auto(ctx.catalog(x), b))
    np.testing.assert_array_equal(parts[0] + parts[1], oracle.count_auto(x, edges, THREADS))


@pytest.mark.parametrize("mode", ["screen", "prune", "check"])
def test_shards_of_the_default_kernel(T, mode):
    """More items than SMs in every shard; with pruning several items a draw, so that the
    last draw of a shard's range is cut short."""
    flags = {"screen": 0, "prune": T.TPCF_F_PRUNE, "check": T.TPCF_F_CHECK_OVERFLOW}[mode]
    n = 60000 if mode != "prune" else 200_000  # (pruned: 44,000 items, 9 or 6 a draw of a half or third)
    d = synth.clustered(n, 256, 0.3, synth.Footprint("sphere"), seed=25)
    r = synth.randoms(n + 30011, synth.Footprint("sphere"), seed=26)
    edges = synth.log_edges(0.02, 6.0, 30)
    full, pairs = _count(T, d, r, edges)
    for world in (2, 3):
        parts = [_count(T, d, r, edges, flags=flags, shard_index=s, shard_count=world) for s in range(world)]
        np.testing.assert_array_equal(np.sum([p[0] for p in parts], axis=0, dtype=np.uint64), full)
        assert sum(p[1] for p in parts) == pairs


@pytest.mark.parametrize("flags", [0, 0x10])
def test_shards_of_the_default_kernel_against_the_oracle(T, flags):
    w = synth.octant_small(seed=6, n=6001)
    want = np.stack([oracle.count_auto(w.data, w.edges, THREADS), oracle.count_cross(w.data, w.rand, w.edges, THREADS),
                     oracle.count_auto(w.rand, w.edges, THREADS)])
    parts = [_count(T, w.data, w.rand, w.edges, flags=flags, shard_index=s, shard_count=3)[0] for s in range(3)]
    np.testing.assert_array_equal(np.sum(parts, axis=0, dtype=np.uint64), want)


def test_shards_in_3d(T):
    d, r = synth.box_clustered(30011, 64, 0.5, 100.0, 7), synth.box_points(20001, 100.0, 8)
    edges = synth.log_edges_r(0.3, 12.0, 17)
    want = [oracle.count_auto(d, edges, THREADS, euclid=True), oracle.count_cross(d, r, edges, THREADS, euclid=True),
            oracle.count_auto(r, edges, THREADS, euclid=True)]
    parts = []
    for s in range(3):
        with T.Context(shard_index=s, shard_count=3) as ctx:
            parts.append(np.stack(ctx.count_all(ctx.catalog3d(d), ctx.catalog3d(r), ctx.bins3d(edges))))
    np.testing.assert_array_equal(np.sum(parts, axis=0, dtype=np.uint64), np.stack(want))
