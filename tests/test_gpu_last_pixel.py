"""Variant (c) on the last pixel of the largest sensors (pixel id 2^20 - 1), in
components long enough that every index modulo the tables' range occurs there."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from gpu_helpers import check_against_oracle  # noqa: E402


@pytest.mark.parametrize("w,h", [(1024, 1024), (65536, 16), (16, 65536)])
@pytest.mark.parametrize("dt", [37, 300, 700])
def test_one_pixel(w, h, dt):
    n = 9000
    hits = oracle.make_hits(np.full(n, w - 1), np.full(n, h - 1), np.arange(n), 1 + np.arange(n) % 7)
    check_against_oracle(hits, w, h, dt, "static")


@pytest.mark.parametrize("seed", range(4))
def test_corner(seed):
    rng = np.random.default_rng(seed)
    n = 20_000
    hits = oracle.make_hits(1022 + rng.integers(0, 2, n), 1022 + rng.integers(0, 2, n), np.arange(n) + 5,
                            rng.integers(1, 50, n))
    check_against_oracle(hits, 1024, 1024, 150 + 200 * seed, "static")
