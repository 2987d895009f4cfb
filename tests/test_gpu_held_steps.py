"""Steps of one context after one that the arrival-order path could not be used
for: the next ones start on the time-sorted path, whatever they hold, and give
the oracle's clusters all the same."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2412_11809_gb300 import Clusterer, TpcError, batch_flush  # noqa: E402
from gpu_helpers import assert_features_equal  # noqa: E402

N = 70_001


def _hits(kind, seed, t0=0, n=N):
    """ordered, shuffled over 2000 or 9000 positions, one hit 12,000 positions late, in no order, or
    dense (no tile holds the hits within dt)."""
    rng = np.random.default_rng(seed)
    toa = t0 + np.arange(n) * 4 // (32 if kind == "dense" else 1)
    hits = oracle.make_hits(rng.integers(0, 256, n), rng.integers(0, 256, n), toa, rng.integers(1, 50, n))
    at = np.arange(n, dtype=float)
    if kind == "late":
        at[20_000] += 12_000.5
    elif kind == "unordered":
        at = rng.permutation(n)
    elif isinstance(kind, int):
        at += rng.integers(0, kind + 1, n)
    return hits[np.argsort(at, kind="stable")]


def _check(c, hits, base, dt):
    want = oracle.labels(hits, 256, 256, dt)
    np.testing.assert_array_equal(c.labels() - np.uint64(base), want)
    rec = c.features()
    rec["label"] -= np.uint64(base)
    assert_features_equal(rec, oracle.features(hits, want))


@pytest.mark.parametrize("kinds", [
    ["unordered", 0, 0, 2000], [9000, "dense", 0, 9000, 0, 0, 0], ["late"] * 6 + [0] * 10,
    [0, "dense", "unordered", 2000, "late", "dense"]])
def test_flushes(kinds):
    with Clusterer(256, 256, 200) as c:
        base = 0
        for k, kind in enumerate(kinds):
            hits = _hits(kind, k, 2**40 * (k % 3))
            c.push(hits)
            c.flush()
            _check(c, hits, base, 200)
            base += len(hits)


def test_small_and_batched_steps_between():
    """Steps of at most 65,536 hits and batches led by the context do not mix with what it holds."""
    with Clusterer(256, 256, 200) as a, Clusterer(256, 256, 200) as b:
        base = {a: 0, b: 0}
        for k, kind in enumerate(["unordered", "late", 0, 0]):
            for n, ctxs in ((N, [a]), (5000, [a]), (N, [a, b])):
                all_hits = [_hits(kind if i == 0 else 0, 10 * k + i, n=n) if n > 30_000 else _hits(0, k, n=n)
                            for i in range(len(ctxs))]
                for c, h in zip(ctxs, all_hits):
                    c.push(h)
                if len(ctxs) > 1:
                    batch_flush(ctxs)
                else:
                    a.flush()
                for c, h in zip(ctxs, all_hits):
                    _check(c, h, base[c], 200)
                    base[c] += len(h)


def test_growing_steps():
    """The arrays grow between the steps, and what the context holds moves along."""
    with Clusterer(256, 256, 200) as c:
        base = 0
        for k, n in enumerate([N, 150_000, 90_000, 400_000, 900_000]):
            hits = _hits("unordered" if k < 3 else 0, k, n=n)
            c.push(hits)
            c.flush()
            _check(c, hits, base, 200)
            base += n


def test_errors_in_held_steps():
    """A hit outside the sensor is reported by a step that starts on the time-sorted path."""
    with Clusterer(256, 256, 200) as c:
        for kind in ("unordered", "unordered"):
            c.push(_hits(kind, 1))
            c.flush()
            c.sync()
        bad = _hits(0, 2)
        bad["x"][N // 2] = 256
        c.push(bad)
        c.flush()
        with pytest.raises(TpcError) as e:
            c.sync()
        assert e.value.name == "TPC_ERR_RANGE"


def test_streaming():
    """A stream whose disorder grows beyond the tiles' margins and shrinks again."""
    n = 100_000
    parts = [_hits(kind, k, 4 * n * k, n) for k, kind in enumerate([0, 9000, 0, 0, 2000, 0])]
    hits = np.concatenate(parts)
    want = oracle.labels(hits, 256, 256, 200)
    got = np.empty(len(hits), dtype=np.uint64)
    with Clusterer(256, 256, 200, max_disorder=80_000) as c:
        for p in parts + [None]:
            if p is None:
                c.flush()
            else:
                c.push(p)
            lab, idx = c.labels(with_indices=True)
            got[idx.astype(np.int64)] = lab
    np.testing.assert_array_equal(got, want)
