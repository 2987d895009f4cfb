"""The (c) sweeps at the sizes where they change (registers, table, window) and
where a window moves on, against the oracle: one component of n hits each."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from gpu_helpers import check_against_oracle  # noqa: E402


@pytest.mark.parametrize("n", [2, 31, 32, 33, 64, 65, 255, 256, 257, 511, 512, 513, 959, 960, 961, 991, 992, 1024, 1025,
                               2047, 2048, 4097, 9001])
@pytest.mark.parametrize("dt", [6, 40])
def test_one_component(n, dt):
    rng = np.random.default_rng(n * 7 + dt)
    hits = oracle.make_hits(rng.integers(0, 5, n), rng.integers(0, 4, n), np.sort(rng.integers(0, n, n)),
                            rng.integers(1, 50, n))
    check_against_oracle(hits, 5, 4, dt, "static")


@pytest.mark.parametrize("within", [900, 1000, 1100])
def test_window_at_its_limit(within):
    """About `within` hits within dt of each other, the window's 960 among them."""
    rng = np.random.default_rng(within)
    n = 5000
    hits = oracle.make_hits(rng.integers(0, 30, n), rng.integers(0, 30, n), np.arange(n) * 3, rng.integers(1, 50, n))
    check_against_oracle(hits, 30, 30, 3 * within, "static")


def test_many_components_of_all_sizes():
    rng = np.random.default_rng(2)
    parts, t = [], 0
    for size in [1, 2, 3, 33, 512, 513, 700, 1500, 2300] * 12:
        x0, y0 = rng.integers(0, 440), rng.integers(0, 500)
        parts.append(np.stack([x0 + rng.integers(0, 5, size), y0 + rng.integers(0, 4, size),
                               t + np.sort(rng.integers(0, max(1, size // 2), size))]))
        t += 300
    x, y, toa = np.concatenate(parts, 1)
    hits = oracle.make_hits(x, y, toa, rng.integers(1, 50, len(x)))
    check_against_oracle(hits[rng.permutation(len(hits))], 448, 512, 25, "static")
