"""The arrival-order path (variant (a), one-shot and streaming) at the edges of
its tiles, its cell grid and its rules, against the oracle: labels and integer
features exact, centroids within the fp32 bound of the other parity tests."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2412_11809_gb300 import Clusterer  # noqa: E402
from gpu_helpers import check_against_oracle  # noqa: E402

SMALL = 65536   # the largest step without a time-sorted path behind it


@pytest.mark.parametrize("n", [1, 31, 4095, 4096, 4097, SMALL - 1, SMALL, SMALL + 1, 73_729, 200_003])
def test_sizes(n):
    hits, _ = synth.cfg1(scale=n / (64 * 2**20), seed=n % 97)
    check_against_oracle(hits[:n], 256, 256, 128)


# one word per row, its border columns; rows sharing cells; one row for all; 16 bands' worth of rows
@pytest.mark.parametrize("w,h", [(1, 1), (1, 9000), (29, 7), (30, 30), (31, 5), (60, 61), (61, 300), (448, 512),
                                 (1024, 1024), (16, 65536), (65536, 16)])
@pytest.mark.parametrize("n", [30_000, 100_001])
def test_sensors(w, h, n):
    hits, _ = synth.generate(w, h, n, w + h + n, hit_rate_hz=40e6, track_frac=0.2, dead_time=True)
    check_against_oracle(hits, w, h, 128)


# wider than the margins (far rounds), wider than those (time-sorted path), none at all
@pytest.mark.parametrize("window", [1, 1000, 2000, 4000, 9000])
def test_disorder(window):
    hits, _ = synth.generate(256, 256, 150_000, window, hit_rate_hz=40e6, track_frac=0.2, dead_time=True,
                             shuffle_window=window)
    check_against_oracle(hits, 256, 256, 128)


@pytest.mark.parametrize("n", [50_000, 130_000])
@pytest.mark.parametrize("order", ["random", "reversed"])
def test_no_order(n, order):
    hits, _ = synth.cfg1(scale=n / (64 * 2**20), seed=5)
    hits = hits[::-1].copy() if order == "reversed" else hits[np.random.default_rng(1).permutation(len(hits))]
    check_against_oracle(hits, 256, 256, 128)


# a tile holds fewer hits than dt spans at 2.5 Ghits/s and dt 384 and beyond
@pytest.mark.parametrize("dt", [0, 1, 384, 2000, 2**27, 2**40])
def test_time_windows(dt):
    hits, _ = synth.cfg4(scale=120_000 / (512 * 2**20), seed=8)
    check_against_oracle(hits, 448, 512, dt)


@pytest.mark.parametrize("n", [9_000, 70_000])
def test_piles(n):
    """Many hits on few pixels, all within dt or spread over a few dt: long lists per cell."""
    rng = np.random.default_rng(n)
    hits = oracle.make_hits(rng.integers(100, 103, n), rng.integers(50, 53, n),
                            np.sort(rng.integers(0, 40 * n, n)), rng.integers(1, 100, n))
    check_against_oracle(hits, 256, 256, 128)


def test_one_instant():
    rng = np.random.default_rng(3)
    n = 20_000
    hits = oracle.make_hits(rng.integers(0, 256, n), rng.integers(0, 256, n), np.full(n, 12345),
                            rng.integers(1, 100, n))
    check_against_oracle(hits, 256, 256, 128)


@pytest.mark.parametrize("n", [3_000, 80_000])
def test_lone_hits(n):
    """Every hit a cluster of its own: as many clusters as hits in every tile."""
    k = np.arange(n)
    hits = oracle.make_hits((k * 37) % 256, (k * 91 // 7) % 256, 1000 + 200 * k, 1 + k % 5)
    check_against_oracle(hits, 256, 256, 0)


@pytest.mark.parametrize("n", [5_000, 70_000])
def test_largest_sums(n):
    """ToT 65535 at high columns: the tile's moments carry beyond 32 bits."""
    rng = np.random.default_rng(n)
    hits = oracle.make_hits(65530 + rng.integers(0, 6, n), rng.integers(0, 2, n), 10 * np.arange(n),
                            np.full(n, 65535))
    check_against_oracle(hits, 65536, 16, 128)


@pytest.mark.parametrize("n", [4_000, 90_000])
def test_long_spans(n):
    """ToAs up to 2^32 - 1 ticks apart, the first hit first, last or in the middle."""
    rng = np.random.default_rng(n)
    toa = np.sort(np.concatenate([rng.integers(0, 4000, n // 2), 2**32 - 1 - rng.integers(0, 4000, n - n // 2)]))
    x, y = rng.integers(0, 20, n), rng.integers(0, 20, n)
    for shift in (0, n // 2, n - 1):
        check_against_oracle(oracle.make_hits(x, y, np.roll(toa, shift), 1 + x), 256, 256, 128)


def test_stream_across_both_forms():
    """Streaming steps below and above the small step's size give the oracle's clusters."""
    hits, t = synth.generate(256, 256, 300_000, 12, hit_rate_hz=40e6, track_frac=0.2, dead_time=True)
    want = oracle.labels(hits, 256, 256, 128)
    got = np.empty(len(hits), dtype=np.uint64)
    with Clusterer(256, 256, 128, max_disorder=t) as c:
        a = 0
        for m in (20_000, 90_000, 1, 40_000, 149_999):
            c.push(hits[a:a + m])
            a += m
            lab, idx = c.labels(with_indices=True)
            got[idx.astype(np.int64)] = lab
        c.flush()
        lab, idx = c.labels(with_indices=True)
        got[idx.astype(np.int64)] = lab
    np.testing.assert_array_equal(got, want)
