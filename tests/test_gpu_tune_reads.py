"""The tuner times only choices that the batch's step reads."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2412_11809_gb300 import Clusterer, tune_batch  # noqa: E402

READ = 1 + 3 + 3 + 3 + 3 + 1    # the defaults; link, acc, out CTAs, general_link, order
SORTED = 2 + 2                  # sort CTAs, span


@pytest.mark.parametrize("order", ["shuffled", "random"])
def test_choices(order):
    hits, _ = synth.generate(256, 256, 200_000, 5, hit_rate_hz=40e6, track_frac=0.2, dead_time=True)
    if order == "random":   # in no order: the time-sorted path
        hits = hits[np.random.default_rng(1).permutation(len(hits))]
    with Clusterer(256, 256, 128) as c:
        c.push(hits)
        rep = tune_batch([c])
        got = rep.chosen.as_dict()
        if order == "random":
            assert rep.trials >= READ + SORTED
        elif got["general_link"] == 0:   # (a choice that gets worse and better again is timed twice)
            assert READ <= rep.trials < 2 * (READ + SORTED) - 1
            assert got["ctas_sort"] == 0 and got["acc_span"] == 1024
        c.flush()
        np.testing.assert_array_equal(c.labels(), oracle.labels(hits, 256, 256, 128))
