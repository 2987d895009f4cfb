"""Tiles taken in parts whose hits arrive late by more than the positions read at
once: all parts of a tile have to read the same ones.  Against the oracle, with
the kernels that ran."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2412_11809_gb300 import Clusterer  # noqa: E402
from gpu_helpers import check_against_oracle  # noqa: E402

TILE = 4096


def _kernels(hits, dt):
    with Clusterer(448, 512, dt) as c:
        c.push(hits)
        return {name for name, _ in c.profile_flush()}


def _moved(hits, moves):
    """Hits in the order given by their index, those of `moves` just before or after a position."""
    at = np.arange(len(hits), dtype=float)
    for i, p in moves.items():
        at[i] = p + (0.5 if p > i else -0.5)
    return hits[np.argsort(at, kind="stable")]


def _stream(n, toa, seed):
    """Hits left of column 440."""
    rng = np.random.default_rng(seed)
    return oracle.make_hits(rng.integers(0, 440, n), rng.integers(0, 512, n), toa, rng.integers(1, 50, n))


@pytest.mark.parametrize("late", [600, 2600])
def test_late_hit_of_an_earlier_part(late):
    """Of one tile's hits, one of the first half of its time (at TILE + 1820 of its index) arrives 2248
    positions behind the tile; another, of the first half or of the second, 2028 behind, so that only
    the part that owns it has a reason of its own to read on.  The late one's neighbour is in the
    second half."""
    n, j = 90_000, 8 * TILE
    hits = _stream(n, 2**29 + np.arange(n) // 4, late)
    hits["x"][[j + 1820, j + 2600]], hits["y"][[j + 1820, j + 2600]] = 445, [100, 101]
    hits = _moved(hits, {j + late: j + TILE + 2028, j + 1820: j + TILE + 2248})
    check_against_oracle(hits, 448, 512, 700)
    ran = _kernels(hits, 700)
    assert "k_arrival_tile_parts" in ran and "k_tile_sort" not in ran


@pytest.mark.parametrize("size", [64, 250, 600])
@pytest.mark.parametrize("delay", [-5000, -2500, 2100, 3000, 5000])
def test_late_blocks(size, delay):
    """Blocks of consecutive hits that arrive late or early by up to 5000 positions, one to each
    20,000, dt over 2000 hits.  (A block of 600 can hold most of the hits that a cut between two tiles
    is taken from, and the tiles then are in no order.)"""
    n = 90_001
    hits = _stream(n, np.arange(n), size + abs(delay))
    moves = {a + k: a + k + delay for a in range(8_000, n - 8_000, 20_000) for k in range(size)}
    hits = _moved(hits, moves)
    check_against_oracle(hits, 448, 512, 2000)
    assert size == 600 or "k_arrival_tile_parts" in _kernels(hits, 2000)


@pytest.mark.parametrize("reach", [1700, 2600])
@pytest.mark.parametrize("disorder", [2500, 4000, 6000])
def test_wide_disorder(reach, disorder):
    """dt over more hits than a tile holds beside its own, in a stream shuffled over more than the margin."""
    n = 80_001
    hits = _stream(n, np.arange(n), reach + disorder)
    hits = hits[np.argsort(np.arange(n) + np.random.default_rng(disorder).integers(0, disorder + 1, n), kind="stable")]
    check_against_oracle(hits, 448, 512, reach)
