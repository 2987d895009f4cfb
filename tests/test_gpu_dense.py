"""Tiles with more hits than one holds at once (a time window that reaches back
over many hits): in parts, from none to all of a step's tiles, and beyond what
parts can take, against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from gpu_helpers import check_against_oracle  # noqa: E402


def _hits(n, toa, disorder, seed):
    rng = np.random.default_rng(seed)
    hits = oracle.make_hits(rng.integers(0, 448, n), rng.integers(0, 512, n), toa, rng.integers(1, 50, n))
    return hits[np.argsort(np.arange(n) + rng.integers(0, disorder + 1, n), kind="stable")]


@pytest.mark.parametrize("reach", [1000, 1400, 1530, 1550, 1700, 2040, 2060, 2600, 4090, 5000])
@pytest.mark.parametrize("disorder", [0, 900])
def test_reach(reach, disorder):
    """dt reaches back over `reach` hits (a tile owns 4096 and holds 5632)."""
    n = 80_001
    check_against_oracle(_hits(n, np.arange(n), disorder, reach), 448, 512, reach, "local")


@pytest.mark.parametrize("burst", [6_000, 9_000, 30_000])
def test_bursts(burst):
    """A sparse stream with dense stretches: some tiles in parts, others not."""
    gaps = np.full(120_000, 40)
    gaps[30_000:30_000 + burst] = 1
    gaps[90_000:90_000 + burst // 2] = 2
    check_against_oracle(_hits(len(gaps), np.cumsum(gaps), 500, burst), 448, 512, 1800, "local")
