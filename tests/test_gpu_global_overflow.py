"""Variant (b) on streams that leave more edges open than their list holds: full
rounds until it fits, the features once, and the next steps of the context."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2412_11809_gb300 import Clusterer  # noqa: E402
from gpu_helpers import assert_features_equal  # noqa: E402


def _hits(n, gap, seed):
    """Events of one to eight hits on 24 x 24 pixels, `gap` ticks apart: every pixel has a latest hit."""
    rng = np.random.default_rng(seed)
    ev = np.sort(rng.integers(0, n // 4, n))
    x0, y0 = rng.integers(0, 22, n // 4), rng.integers(0, 22, n // 4)
    return oracle.make_hits(x0[ev] + rng.integers(0, 3, n), y0[ev] + rng.integers(0, 3, n),
                            2**31 + ev * gap + rng.integers(0, 30, n), rng.integers(1, 50, n))


@pytest.mark.parametrize("gap", [40, 300, 3000])
@pytest.mark.parametrize("n", [3000, 60_000, 200_000])
def test_sparse(n, gap):
    with Clusterer(64, 64, 100, "global") as c:
        base, full = 0, 0
        for k, g in enumerate([gap, gap, 2, gap]):
            hits = _hits(n, g, 5 * k + n)
            c.push(hits)
            c.flush()
            want = oracle.labels(hits, 64, 64, 100, "global")
            np.testing.assert_array_equal(c.labels() - np.uint64(base), want)
            rec = c.features()
            rec["label"] -= np.uint64(base)
            assert_features_equal(rec, oracle.features(hits, want))
            full = max(full, c.variant_stats()["full_rounds"])
            base += n
        if gap == 40:
            assert full > 1   # (a list holds two edges per position; most hits leave more, and some merge)
