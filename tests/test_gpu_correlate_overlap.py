"""One-call correlation, whose two preparations and bins overlap: errors come
in the order data, randoms, bins; every failing allocation is reported and the
context stays usable; several threads with their own streams."""
import os
import threading

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


def _data(n, seed):
    d, r = synth.clustered(n, 8, 0.5, seed=seed), synth.randoms(2 * n + 1, seed=seed + 1)
    e = synth.linear_edges(0.0, 3.0, 12)
    return d, r, e, (oracle.count_auto(d, e, THREADS), oracle.count_cross(d, r, e, THREADS),
                     oracle.count_auto(r, e, THREADS))


@pytest.mark.parametrize("bad", ["d", "r", "dr"])
def test_errors_and_after(T, bad):
    d, r, e, want = _data(777, 4)
    d2, r2 = d.copy(), r.copy()
    if "d" in bad:
        d2[5] *= 2.0
    if "r" in bad:
        r2[-1, 0] = np.nan
    with T.Context() as ctx:
        with pytest.raises(Exception, match="unit vector"):
            ctx.correlate(d2, r2, e)
        for g, o in zip(ctx.correlate(d, r, e), want):
            np.testing.assert_array_equal(g, o)


def test_failing_allocations(T):
    d, r, e, want = _data(300, 9)
    with T.Context() as ctx:
        failed = 0
        for k in range(6):
            T.load().tpcf_debug_fail_alloc_after(k)
            try:
                ctx.correlate(d, r, e)
            except Exception:
                failed += 1
            finally:
                T.load().tpcf_debug_fail_alloc_after(-1)
        assert failed == 3  # two catalogs and the bins
        for g, o in zip(ctx.correlate(d, r, e), want):
            np.testing.assert_array_equal(g, o)


def test_threads(T):
    import torch
    sets = [_data(500 + 301 * k, 20 + k) for k in range(4)]
    out = [None] * 4
    with T.Context() as ctx:
        def work(k):
            s = torch.cuda.Stream()
            out[k] = [ctx.correlate(*sets[k][:3], stream=s.cuda_stream) for _ in range(5)]
        ts = [threading.Thread(target=work, args=(k,)) for k in range(4)]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
    for k in range(4):
        assert out[k] is not None
        for res in out[k]:
            for g, o in zip(res, sets[k][3]):
                np.testing.assert_array_equal(g, o)
