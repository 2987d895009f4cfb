"""Small steps whose tiles of positions are not done: no order, more hits within
dt than a tile holds, many hits on one pixel.  The step is sorted by pixel and
time and joined hit by hit; against the oracle, with every entry that takes
small steps."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2412_11809_gb300 import Clusterer  # noqa: E402
from gpu_helpers import check_against_oracle  # noqa: E402


def _hits(toa, w, h, seed, tot=50):
    rng = np.random.default_rng(seed)
    n = len(toa)
    return oracle.make_hits(rng.integers(0, w, n), rng.integers(0, h, n), toa, rng.integers(1, tot, n))


@pytest.mark.parametrize("n", [4097, 8192, 40_961, 65_535, 65_536])
@pytest.mark.parametrize("dt", [0, 60, 3000, 2**20, 2**31])
def test_no_order(n, dt):
    """From hits that join nothing to a dt over the whole step."""
    rng = np.random.default_rng(n)
    step = 1 if dt < 2**20 else 2**15
    check_against_oracle(_hits(rng.permutation(n) * step + 2**33, 256, 256, n), 256, 256, dt, "local")


@pytest.mark.parametrize("rate", [2, 16, 64])
@pytest.mark.parametrize("disorder", [0, 1000, 9000])
def test_dense(rate, disorder):
    """Up to 24,000 hits within dt."""
    n = 50_000
    at = np.arange(n) + np.random.default_rng(rate).integers(0, disorder + 1, n)
    hits = _hits(2**29 + np.arange(n) // rate, 448, 512, rate + disorder)
    check_against_oracle(hits[np.argsort(at, kind="stable")], 448, 512, 384, "local")


@pytest.mark.parametrize("n", [1500, 5000, 65_536])
@pytest.mark.parametrize("pixels", [1, 2, 5])
def test_piles(n, pixels):
    """All hits on a few pixels; dt within a pixel's gaps, so that some join and some do not."""
    rng = np.random.default_rng(n + pixels)
    toa = np.cumsum(rng.integers(0, 40, n))
    hits = oracle.make_hits(100 + rng.integers(0, pixels, n), np.full(n, 7), toa, rng.integers(1, 50, n))
    check_against_oracle(hits, 256, 256, 30 * pixels, "local")
    check_against_oracle(hits[rng.permutation(n)], 256, 256, 30 * pixels, "local")


@pytest.mark.parametrize("w,h", [(1, 1), (1, 65536), (65536, 1), (1024, 1024), (16, 65536), (65536, 16), (3, 2)])
def test_sensors(w, h):
    rng = np.random.default_rng(w + h)
    n = 9000
    toa = rng.permutation(n) * 3
    hits = oracle.make_hits(w - 1 - rng.integers(0, min(w, 20), n), h - 1 - rng.integers(0, min(h, 20), n), toa,
                            rng.integers(1, 50, n))
    check_against_oracle(hits, w, h, 100, "local")


def test_equal_times_keep_their_order():
    """One instant: every hit's label and ties decided by input order."""
    hits = _hits(np.full(30_000, 77), 300, 300, 1)
    check_against_oracle(hits, 300, 300, 0, "local")


def test_largest_sums():
    """One cluster of 65,536 hits of ToT 65,535 at high columns."""
    n = 65_536
    rng = np.random.default_rng(4)
    hits = oracle.make_hits(np.full(n, 65_535), rng.integers(0, 2, n), rng.permutation(n), np.full(n, 65_535))
    check_against_oracle(hits, 65536, 16, 500, "local")


def test_streaming_and_static():
    """The same through a streaming context (open hits carried) and the allocation-free call."""
    rng = np.random.default_rng(9)
    n, parts = 30_000, 4
    hits = _hits(2**30 + np.arange(n * parts) // 8, 256, 256, 5)
    hits = hits[np.argsort(np.arange(n * parts) + rng.integers(0, 8000, n * parts), kind="stable")]
    want = oracle.labels(hits, 256, 256, 384)
    got = np.empty(len(hits), dtype=np.uint64)
    with Clusterer(256, 256, 384, max_disorder=1200) as c:
        for k in range(parts + 1):
            if k < parts:
                c.push(hits[k * n:(k + 1) * n])
            else:
                c.flush()
            lab, idx = c.labels(with_indices=True)
            got[idx.astype(np.int64)] = lab
    np.testing.assert_array_equal(got, want)
    from paper_2412_11809_gb300 import binding
    lib = binding.load_library()
    part = hits[:n]
    want = oracle.labels(part, 256, 256, 384)
    d = torch.from_numpy(part.view(np.uint8).reshape(-1, 16)).cuda()
    labels = torch.empty(n, dtype=torch.int64, device="cuda")
    records = torch.empty((n, 40), dtype=torch.uint8, device="cuda")
    counts = torch.empty(2, dtype=torch.int64, device="cuda")
    rc = lib.tpc_cluster_static(d.data_ptr(), n, 256, 256, 384, labels.data_ptr(), records.data_ptr(), n,
                                counts.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    assert counts.cpu().tolist() == [len(np.unique(want)), 0]
    np.testing.assert_array_equal(labels.cpu().numpy().astype(np.uint64), want)
