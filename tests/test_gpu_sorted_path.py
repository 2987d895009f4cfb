"""The time-sorted path on streams and choices that the arrival-order path now
takes by default: merges of tiles that interleave over one and both bands, the
general sort behind them, every span of the feature kernel."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2412_11809_gb300 import Clusterer  # noqa: E402
from gpu_helpers import assert_features_equal, check_against_oracle  # noqa: E402


def _hits(window, n, seed=0):
    return synth.generate(256, 256, n, 40 + window + seed, hit_rate_hz=40e6, track_frac=0.2, dead_time=True,
                          shuffle_window=window)[0]


@pytest.mark.parametrize("window", [1000, 2400, 5000])
@pytest.mark.parametrize("variant", ["global", "static"])
def test_variants(window, variant):
    check_against_oracle(_hits(window, 150_000), 256, 256, synth.DT_200NS, variant)


@pytest.mark.parametrize("window", [1000, 2400, 5000])
@pytest.mark.parametrize("span", [512, 1024, 2048])
@pytest.mark.parametrize("variant", ["local", "static"])
def test_spans(window, span, variant):
    hits = _hits(window, 200_000, span)
    want = oracle.labels(hits, 256, 256, synth.DT_200NS, variant)
    with Clusterer(256, 256, synth.DT_200NS, variant) as c:
        c.set_tuning({"acc_span": span, "general_link": 3})   # general_link: time-sorted from the start
        c.push(hits)
        names = {k for k, _ in c.profile_flush()}
        assert "k_accumulate" in names and "k_arrival_tile" not in names
        np.testing.assert_array_equal(c.labels(), want)
        assert_features_equal(c.features(), oracle.features(hits, want))


@pytest.mark.parametrize("window", [1000, 2400, 5000])
def test_table_link(window):
    """Behind an arrival-order attempt: hits no two of which are alone, more of them within dt than a
    tile's parts hold, then streams of every width in the steps the context holds on that path."""
    rng = np.random.default_rng(window)
    n = 100_000
    dense = oracle.make_hits(rng.integers(0, 256, n), rng.integers(0, 256, n), np.arange(n) // 64, rng.integers(1, 50, n))
    with Clusterer(256, 256, synth.DT_200NS) as c:
        base = 0
        for k, hits in enumerate([dense, _hits(window, 150_000, 1), _hits(window, 150_000, 2)]):
            want = oracle.labels(hits, 256, 256, synth.DT_200NS)
            c.push(hits)
            names = {name for name, _ in c.profile_flush()}
            assert "k_tile_link_table" in names and "k_arrival_labels" not in names
            np.testing.assert_array_equal(c.labels() - np.uint64(base), want)
            rec = c.features()
            rec["label"] -= np.uint64(base)
            assert_features_equal(rec, oracle.features(hits, want))
            base += len(hits)
