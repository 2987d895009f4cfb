"""Small steps on a device that cannot hold their cluster of CTAs (part of a GPU):
the same results by the other paths."""
import ctypes

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2412_11809_gb300 import CLUSTER_DTYPE, Clusterer, binding  # noqa: E402
from gpu_helpers import assert_features_equal  # noqa: E402


@pytest.fixture(scope="module")
def lib():
    lib = binding.load_library()
    lib.tpc_internal_static.argtypes = lib.tpc_cluster_static.argtypes + [ctypes.c_int]
    lib.tpc_internal_most_ctas.argtypes = [ctypes.c_void_p, ctypes.c_int]
    return lib


def _hits(n, order, seed=3):
    hits, _ = synth.generate(256, 256, n, seed, hit_rate_hz=40e6, track_frac=0.2, dead_time=True)
    return hits if order == "shuffled" else hits[np.random.default_rng(seed).permutation(n)]


@pytest.mark.parametrize("most", [0, 1, 4, 16])
@pytest.mark.parametrize("n", [1, 4097, 30_000, 65_536])
@pytest.mark.parametrize("order", ["shuffled", "random"])
def test_static(lib, most, n, order):
    hits = _hits(n, order)
    d = torch.from_numpy(hits.view(np.uint8).reshape(-1, 16)).cuda()
    labels = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    records = torch.zeros((n, CLUSTER_DTYPE.itemsize), dtype=torch.uint8, device="cuda")
    counts = torch.full((2,), -1, dtype=torch.int64, device="cuda")
    want = oracle.labels(hits, 256, 256, 128)
    for cap in (n, 0):   # with records, and labels alone
        rc = lib.tpc_internal_static(d.data_ptr(), n, 256, 256, 128, labels.data_ptr(),
                                     records.data_ptr() if cap else None, cap, counts.data_ptr(),
                                     torch.cuda.current_stream().cuda_stream, most)
        assert rc == 0
        assert counts.cpu().tolist() == [len(np.unique(want)), 0]
        np.testing.assert_array_equal(labels.cpu().numpy().astype(np.uint64), want)
    rec = records.cpu().numpy().reshape(-1).view(CLUSTER_DTYPE)[: len(np.unique(want))]
    assert_features_equal(rec, oracle.features(hits, want))


@pytest.mark.parametrize("order", ["shuffled", "random"])
def test_context(lib, order):
    """Flushes, and a stream of steps of all sizes, none of them in one launch."""
    with Clusterer(256, 256, 128) as c:
        assert lib.tpc_internal_most_ctas(c._h, 8) == 0
        base = 0
        for n in (1, 5000, 65_536):
            hits = _hits(n, order, n % 97)
            want = oracle.labels(hits, 256, 256, 128)
            c.push(hits)
            names = {k for k, _ in c.profile_flush()}
            assert "k_arrival_step" not in names and "k_arrival_tile" in names
            np.testing.assert_array_equal(c.labels() - np.uint64(base), want)
            rec = c.features()
            rec["label"] -= np.uint64(base)
            assert_features_equal(rec, oracle.features(hits, want))
            base += n
    hits, t = synth.generate(256, 256, 60_000, 12, hit_rate_hz=40e6, track_frac=0.2, dead_time=True)
    want = oracle.labels(hits, 256, 256, 128)
    got = np.empty(len(hits), dtype=np.uint64)
    with Clusterer(256, 256, 128, max_disorder=t) as c:
        assert lib.tpc_internal_most_ctas(c._h, 0) == 0
        a = 0
        for m in (1, 20_000, 7, 39_992, 0):
            if m:
                c.push(hits[a:a + m])
            else:
                c.flush()
            a += m
            lab, idx = c.labels(with_indices=True)
            got[idx.astype(np.int64)] = lab
    np.testing.assert_array_equal(got, want)
