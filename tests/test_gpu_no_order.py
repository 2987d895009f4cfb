"""Small steps without order in time, whose tiles are intervals of ToAs, at the
edges of a tile and of a step, and where those hold too many hits, against the
oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from gpu_helpers import check_against_oracle  # noqa: E402


def _hits(toa, w, h, seed):
    rng = np.random.default_rng(seed)
    n = len(toa)
    return oracle.make_hits(rng.integers(0, w, n), rng.integers(0, h, n), toa, rng.integers(1, 50, n))


@pytest.mark.parametrize("n", [4097, 8192, 8193, 30_001, 65_535, 65_536])
@pytest.mark.parametrize("dt", [0, 40, 900, 1900])
def test_shuffled(n, dt):
    rng = np.random.default_rng(n + dt)
    check_against_oracle(_hits(rng.permutation(n), 448, 512, n), 448, 512, dt, "local")


@pytest.mark.parametrize("n", [9_000, 40_000])
@pytest.mark.parametrize("share", [0.2, 0.6, 1.0])
def test_one_instant_among_others(n, share):
    """A share of the hits at one ToA: more than an interval can hold."""
    rng = np.random.default_rng(int(n * share))
    toa = rng.permutation(n).astype(np.int64) * 3 + 2**40
    toa[: int(n * share)] = 2**40 + n
    check_against_oracle(_hits(rng.permutation(toa), 448, 512, n), 448, 512, 2, "local")


@pytest.mark.parametrize("dt", [2**20, 2**27, 2**31])
def test_far_apart(dt):
    """ToAs over most of 32 bits, keys relative to the smallest one."""
    rng = np.random.default_rng(5)
    check_against_oracle(_hits(rng.integers(0, 2**32 - 2, 12_000) + 7, 448, 512, 3), 448, 512, dt, "local")
