"""Variant (b) where its timelines and its large clusters change: timelines of
every length around powers of two, sensor edges, and one to three clusters that
hold nearly all hits and take turns, against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from gpu_helpers import check_against_oracle  # noqa: E402


@pytest.mark.parametrize("w,h", [(1, 1), (1, 3), (2, 2), (3, 3), (5, 4)])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 127, 1025, 4097])
def test_timelines(w, h, n):
    rng = np.random.default_rng(n * 31 + w)
    hits = oracle.make_hits(rng.integers(0, w, n), rng.integers(0, h, n), np.sort(rng.integers(0, 4 * n, n)),
                            rng.integers(1, 50, n))
    check_against_oracle(hits, w, h, 9, "global")


@pytest.mark.parametrize("clusters,run", [(1, 1), (2, 1), (2, 40), (2, 5000), (3, 700)])
def test_large_clusters_in_turn(clusters, run):
    """Columns far apart, each one cluster, a turn of `run` hits each."""
    n = 40000
    rng = np.random.default_rng(run)
    col = (np.arange(n) // run) % clusters
    hits = oracle.make_hits(10 * col + rng.integers(0, 3, n), rng.integers(0, 3, n), np.arange(n),
                            rng.integers(1, 1000, n))
    check_against_oracle(hits, 40, 8, 3 * run * clusters + 40, "global")
