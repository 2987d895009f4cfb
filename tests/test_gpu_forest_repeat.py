"""tpc_forest of arrival-order steps: the same twice, beside the step's other
results, and in the steps after it; for small steps in and out of order, larger
ones, streams, and one cluster that holds everything."""
import time

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2412_11809_gb300 import Clusterer  # noqa: E402
from test_gpu_forest import check_forest  # noqa: E402


def _hits(n, order, seed):
    hits = synth.generate(256, 256, n, seed, hit_rate_hz=40e6, track_frac=0.2, dead_time=True)[0]
    return hits if order == "shuffled" else hits[np.random.default_rng(seed).permutation(n)]


@pytest.mark.parametrize("order", ["shuffled", "random"])
def test_twice_and_between_steps(order):
    with Clusterer(256, 256, 128) as c:
        base = 0
        for k, n in enumerate([1, 33, 30_000, 200_000, 65_536, 500_000]):
            hits = _hits(n, order if n <= 65_536 else "shuffled", k)
            c.push(hits)
            c.flush()
            want = oracle.labels(hits, 256, 256, 128)
            for _ in range(2):
                parent, pos = c.forest()
                check_forest(hits, parent, pos, want)
                np.testing.assert_array_equal(c.labels() - np.uint64(base), want)
                assert c.counts()[1] == len(np.unique(want)) == len(c.features())
            base += n


def test_one_cluster():
    n = 150_000
    rng = np.random.default_rng(0)
    hits = oracle.make_hits(rng.integers(0, 8, n), rng.integers(0, 8, n), 2**40 + np.arange(n) * 7, np.ones(n, int))
    with Clusterer(256, 256, 2000) as c:
        c.push(hits)
        c.flush()
        check_forest(hits, *c.forest(), oracle.labels(hits, 256, 256, 2000))


def test_stream_goes_on():
    """A forest read after each streaming step changes nothing of the stream."""
    hits, t = synth.generate(256, 256, 400_000, 12, hit_rate_hz=40e6, track_frac=0.2, dead_time=True)
    got = np.empty(len(hits), dtype=np.uint64)
    with Clusterer(256, 256, 128, max_disorder=t) as c:
        a = 0
        for m in (150_000, 20_000, 130_000, 100_000, 0):
            if m:
                c.push(hits[a:a + m])
            else:
                c.flush()
            a += m
            c.forest()
            lab, idx = c.labels(with_indices=True)
            got[idx.astype(np.int64)] = lab
    np.testing.assert_array_equal(got, oracle.labels(hits, 256, 256, 128))


def test_takes_no_longer_than_its_copies_ask_for():
    """4 M hits: 1.7 ms (60 when the order was found on the host, one hit after another)."""
    hits = _hits(4_000_000, "shuffled", 3)
    with Clusterer(256, 256, 128) as c:
        best = 1.0
        for _ in range(3):
            c.push(hits)
            c.flush()
            c.sync()
            t0 = time.perf_counter()
            c.forest()
            best = min(best, time.perf_counter() - t0)
    assert best < 0.03
