"""The work this library is used for, as timed cases.

A case is a dict of plain values.  ``prepare`` makes what a program holds
before the call (a seeded hit stream and, where the interface has one, a
context), ``run`` is one pass through the public entry points and returns
every output whole, ``work`` counts the bytes the path cannot do without, and
``exact`` gives the centroids in 64 bits from a plain clustering in torch.

Interfaces (``call``):

* ``fixed``    ``tpc_cluster_static``: a real-time readout loop that may not
               allocate; device buffers in and out.
* ``oneshot``  ``Clusterer`` on a device tensor, labels returned as a new
               device tensor, records copied into the caller's: the
               interface's plain form.
* ``bound``    ``Clusterer`` writing straight into caller buffers
               (``bind_outputs``): the throughput form.
* ``batch``    ``batch_flush`` over several detectors with bound outputs.
* ``stream``   a streaming ``Clusterer`` fed chunk by chunk from pinned host
               memory, results read back after each chunk into the
               acquisition's pinned arrays, started from a checkpoint.
* ``host``     one-shot from a numpy array, results as numpy arrays.

The number of clusters depends on the stream, so record buffers hold one
record per hit, as a caller who does not know it allocates them; what lies
behind the last record stays zero.

The streams follow the recipe of the benchmark configurations: random-walk
blobs of 1 + Geometric(0.3) pixels, or 80 % such blobs and 20 % straight
tracks of 10 to 300 pixels with dead-time refires, ToT 1 + Exp(40) up to 1023,
ToA jitter of up to 64 ticks, arrival shuffled within 1000 positions.
"""
import math
import random

import numpy as np
import torch

from paper_2412_11809_gb300 import Clusterer, batch_flush
from paper_2412_11809_gb300.binding import CLUSTER_DTYPE, HIT_DTYPE, load_library

TICKS_PER_SECOND = 6.4e8
SHUFFLE = 1000
BLOB_MAX = 24
TRACK_MAX = 300


def _case(name, call, n, width, height, dt, rate, mix=True, variant="local", arrival="shuffled", parts=1):
    """rate: million hits per second (million events for blobs only).  parts:
    detectors of a batch, or hits per chunk of a stream."""
    c = {"call": call, "n": n, "width": width, "height": height, "dt": dt, "rate": rate, "mix": mix,
         "variant": variant, "arrival": arrival, "parts": parts}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a readout loop's smallest batch: the latency of one call
        _case("fixed_1k", "fixed", 1000, 256, 256, 128, 40.0),
        # the largest batch the allocation-free call takes
        _case("fixed_64k", "fixed", 65536, 256, 256, 128, 40.0),
        # a frame-sized batch through the plain interface
        _case("oneshot_100k", "oneshot", 100_003, 256, 256, 128, 40.0),
        # 1 M hits of a photon source: blobs only, at 1 Mevent/s
        _case("oneshot_blobs_1m", "oneshot", 1_000_000, 256, 256, 128, 1.0, mix=False),
        # hits concatenated from several readouts: no arrival order at all
        _case("oneshot_unordered_4m", "oneshot", 4_000_003, 256, 256, 128, 40.0, arrival="unordered"),
        # the library's headline: 64 Mi hits of the 256x256 sensor
        _case("bound_256_64mi", "bound", 64 << 20, 256, 256, 128, 40.0),
        # the large sensor at its full rate
        _case("bound_448x512_32m", "bound", 32_000_001, 448, 512, 128, 2500.0),
        # the other two temporal conditions on the large sensor
        _case("oneshot_global_8m", "oneshot", 8_000_003, 448, 512, 128, 2500.0, variant="global"),
        _case("oneshot_static_8m", "oneshot", 8_000_003, 448, 512, 128, 2500.0, variant="static"),
        # a telescope of 16 detectors of two kinds in one step
        _case("batch_16_40m", "batch", 40_000_000, 0, 0, 128, 40.0, parts=16),
        # an acquisition read out in quarter-million-hit chunks, the last one a sliver
        _case("stream_250k", "stream", 2_000_003, 256, 256, 128, 50.0, parts=250_000),
        # a recorded file clustered from host memory
        _case("host_2m", "host", 2_000_003, 256, 256, 128, 40.0),
    ]


def _log_uniform(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng: random.Random):
    call = rng.choice(["fixed", "oneshot", "oneshot", "oneshot", "bound", "batch", "stream", "host"])
    big = rng.random() < 0.4
    width, height = (448, 512) if big else (256, 256)
    top = 2500.0 if big else 80.0
    rate = float(round(math.exp(rng.uniform(math.log(5.0), math.log(top))), 3))
    dt = rng.choice([128, 128, 384])

    def within(n, r):
        """A step's hits lie within 2^32 ticks (6.7 s): the least rate for n hits."""
        return max(r, math.ceil(n / 6.0e6))

    if call == "fixed":
        return _case(None, call, _log_uniform(rng, 1, 65536), width, height, dt, rate)
    if call == "oneshot":
        variant = rng.choice(["local", "local", "local", "global", "static"])
        arrival = rng.choice(["shuffled"] * 5 + ["unordered"])
        if rng.random() < 0.25:
            return _case(None, call, _log_uniform(rng, 1_000, 8_000_000), 256, 256, dt, 1.0, mix=False,
                         variant=variant, arrival=arrival)
        return _case(None, call, _log_uniform(rng, 1_000, 8_000_000), width, height, dt, rate,
                     variant=variant, arrival=arrival)
    if call == "bound":
        n = _log_uniform(rng, 1_000_000, 32_000_000 if big else 64 << 20)
        return _case(None, call, n, width, height, dt, float(within(n, rate)))
    if call == "batch":
        n = _log_uniform(rng, 100_000, 40_000_000)
        return _case(None, call, n, 0, 0, dt, float(within(n, round(rng.uniform(5.0, 80.0), 3))),
                     parts=rng.randint(2, 16))
    if call == "stream":
        chunk = _log_uniform(rng, 65_536, 1_000_000)
        return _case(None, call, rng.randint(chunk + 1, 6 * chunk), 256, 256, dt, float(round(rng.uniform(5.0, 80.0), 3)),
                     parts=chunk)
    return _case(None, call, _log_uniform(rng, 10_000, 2_000_000), 256, 256, dt, rate if not big else 40.0)


# ---------------------------------------------------------------------------
# inputs


def _prefix_max(x):
    """Running maximum of a 1-D int64 tensor, in two levels."""
    n, cols = x.numel(), 4096
    rows = max(1, -(-n // cols))
    low = torch.iinfo(torch.int64).min
    full = torch.full((rows * cols,), low, dtype=torch.int64, device=x.device)
    full[:n] = x
    m = torch.cummax(full.view(rows, cols), 1).values
    before = torch.full((rows, 1), low, dtype=torch.int64, device=x.device)
    if rows > 1:
        before[1:, 0] = torch.cummax(m[:-1, -1], 0).values
    return torch.maximum(m, before).view(-1)[:n]


def _blobs(gen, count, width, height, device):
    """(event, pixel) of random-walk blobs; pixel = y * width + x."""
    def unit(k):
        return torch.rand(k, generator=gen, device=device)

    size = (1 + torch.floor(torch.log1p(-unit(count)) / math.log(0.7))).clamp_(max=BLOB_MAX).to(torch.int64)
    pix = torch.full((count, BLOB_MAX), -1, dtype=torch.int64, device=device)
    pix[:, 0] = torch.randint(0, width * height, (count,), generator=gen, device=device)
    have = torch.ones(count, dtype=torch.int64, device=device)
    for _ in range(2 * BLOB_MAX):
        act = torch.nonzero(have < size).view(-1)
        if act.numel() == 0:
            break
        m = have[act]
        parent = pix[act, (unit(act.numel()) * m).to(torch.int64).clamp_(max=BLOB_MAX - 1)]
        d = torch.randint(0, 8, (act.numel(),), generator=gen, device=device)
        d = d + (d >= 4)   # the 3x3 neighbourhood without its centre
        x, y = parent % width + d % 3 - 1, parent // width + d // 3 - 1
        new = y * width + x
        ok = (x >= 0) & (x < width) & (y >= 0) & (y < height) & ~(pix[act] == new[:, None]).any(1)
        act, new, m = act[ok], new[ok], m[ok]
        pix[act, m] = new
        have[act] = m + 1
    ev, col = torch.nonzero(pix >= 0, as_tuple=True)
    return ev, pix[ev, col], have


def _tracks(gen, count, width, height, device):
    """(event, pixel, time offset) of straight tracks rastered along their major axis."""
    def unit():
        return torch.rand(count, generator=gen, device=device)

    length = 10 + torch.floor(unit() * (TRACK_MAX - 9))
    theta, g = unit() * math.pi, unit() * 20.0
    c, s = torch.cos(theta), torch.sin(theta)
    major = torch.maximum(c.abs(), s.abs())
    sx, sy = c / major, s / major
    x0, y0 = torch.floor(unit() * width), torch.floor(unit() * height)
    evs, pixs, offs = [], [], []
    k = torch.arange(TRACK_MAX, device=device, dtype=torch.float32)
    for a in range(0, count, 1 << 17):
        b = min(count, a + (1 << 17))
        x = torch.floor(x0[a:b, None] + 0.5 + k * sx[a:b, None])
        y = torch.floor(y0[a:b, None] + 0.5 + k * sy[a:b, None])
        ok = (k < length[a:b, None]) & (x >= 0) & (x < width) & (y >= 0) & (y < height)
        ev, col = torch.nonzero(ok, as_tuple=True)
        evs.append(ev + a)
        pixs.append(y[ev, col].to(torch.int64) * width + x[ev, col].to(torch.int64))
        offs.append(torch.floor(col * g[a + ev]).to(torch.int64))
    return torch.cat(evs), torch.cat(pixs), torch.cat(offs)


def _stream(case, n, width, height, rate, seed):
    """(hits, t): n 16-byte records as an (n, 2) int64 CUDA tensor, and the
    smallest t for which the stream is t-ordered."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) * 1_000_003 + 17)
    target = n + n // 50 + 64
    toas, pixs, total, clock = [], [], 0, 1_000_000 << 12
    while total < target:
        count = int((target - total) / (18.0 if case["mix"] else 3.0)) + 64
        if case["mix"]:
            track = torch.rand(count, generator=gen, device=dev) < 0.2
            where_b, where_t = torch.nonzero(~track).view(-1), torch.nonzero(track).view(-1)
        else:
            where_b, where_t = torch.arange(count, device=dev), torch.empty(0, dtype=torch.int64, device=dev)
        ev, pix, _ = _blobs(gen, where_b.numel(), width, height, dev)
        ev, off = where_b[ev], torch.zeros_like(pix)
        if where_t.numel():
            ev_t, pix_t, off_t = _tracks(gen, where_t.numel(), width, height, dev)
            ev, pix, off = torch.cat([ev, where_t[ev_t]]), torch.cat([pix, pix_t]), torch.cat([off, off_t])
        got = torch.bincount(ev, minlength=count)
        gap = -torch.log1p(-torch.rand(count, generator=gen, device=dev, dtype=torch.float64))
        per_tick = rate * 1e6 / TICKS_PER_SECOND
        gap = gap * (got.clamp(min=1) if case["mix"] else 1) / per_tick
        gap = (gap * 4096).to(torch.int64)   # whole 1/4096 ticks: sums are exact
        begin = clock + torch.cumsum(gap, 0) - gap
        clock = int(begin[-1] + gap[-1])
        toas.append((begin[ev] >> 12) + off + torch.randint(0, 65, (ev.numel(),), generator=gen, device=dev))
        pixs.append(pix)
        total += int(ev.numel())
    toa, pix = torch.cat(toas), torch.cat(pixs)
    toa, order = torch.sort(toa, stable=True)
    toa, pix = toa[:target], pix[order][:target]
    tot = (1 + torch.floor(-40.0 * torch.log1p(-torch.rand(target, generator=gen, device=dev)) + 0.5))
    tot = tot.clamp_(max=1023).to(torch.int64)
    if case["mix"]:   # a pixel still busy with a hit fires again only when it is free
        order = torch.sort(pix, stable=True).indices
        t, p, w = toa[order], pix[order], tot[order]
        spent = torch.cumsum(w, 0) - w
        toa[order] = _prefix_max(t - spent + (p << 40)) - (p << 40) + spent
        toa, order = torch.sort(toa, stable=True)
        pix, tot = pix[order], tot[order]
    toa, pix, tot = toa[:n], pix[:n], tot[:n]
    if case["arrival"] == "unordered":
        order = torch.randperm(n, generator=gen, device=dev)
    else:
        late = torch.arange(n, device=dev) + torch.randint(0, SHUFFLE, (n,), generator=gen, device=dev)
        order = torch.sort(late, stable=True).indices
    toa, pix, tot = toa[order], pix[order], tot[order]
    hits = torch.stack([(pix % width) | (pix // width) << 16 | tot << 32, toa], 1).contiguous()
    t = int((_prefix_max(toa) - toa).max()) + 1
    return hits, t


def _detectors(case):
    """(width, height, hits, rate) per detector of a batch: ten of 16 are
    256x256, the others 448x512, and their loads differ by up to 16 times."""
    k = case["parts"]
    rng = random.Random(case["n"] * 31 + k)
    weight = [math.exp(rng.uniform(0.0, math.log(16.0))) for _ in range(k)]
    total = sum(weight)
    n = [max(1, int(case["n"] * v / total)) for v in weight]
    return [(256, 256, n[i], case["rate"]) if i % 8 < 5 else (448, 512, n[i], case["rate"]) for i in range(k)]


def _buffers(n, host=False):
    """Zeroed labels and records of n hits, on the device or pinned."""
    place = {"pin_memory": True} if host else {"device": "cuda"}
    return (torch.zeros(n, dtype=torch.int64, **place),
            torch.zeros((n, CLUSTER_DTYPE.itemsize), dtype=torch.uint8, **place))


def _bound(width, height, case, hits):
    c = Clusterer(width, height, case["dt"], case["variant"])
    labels, records = _buffers(hits.shape[0])
    c.bind_outputs(labels.data_ptr(), records.data_ptr(), hits.shape[0])
    return {"ctx": c, "hits": hits, "labels": labels, "records": records}


def prepare(case, seed):
    call, w, h, n = case["call"], case["width"], case["height"], case["n"]
    if call == "batch":
        dets = []
        for i, (dw, dh, dn, rate) in enumerate(_detectors(case)):
            dets.append(_bound(dw, dh, case, _stream(case, dn, dw, dh, rate, seed * 64 + i)[0]))
        torch.cuda.synchronize()
        return {"call": call, "dets": dets}
    hits, t = _stream(case, n, w, h, case["rate"], seed)
    state = {"call": call, "case": case, "hits": hits}
    if call == "fixed":
        state["labels"], state["records"] = _buffers(n)
        state["counts"] = torch.zeros(2, dtype=torch.int64, device="cuda")
        state["lib"] = load_library()
    elif call == "oneshot":
        state["records"] = _buffers(n)[1]
        state["ctx"] = Clusterer(w, h, case["dt"], case["variant"])
    elif call == "bound":
        state.update(_bound(w, h, case, hits))
    elif call == "stream":
        pinned = torch.empty(hits.shape, dtype=torch.int64, pin_memory=True)
        state["hits"] = pinned.copy_(hits)
        state["labels"], state["records"] = _buffers(n, host=True)
        state["indices"] = torch.zeros(n, dtype=torch.int64, pin_memory=True)
        state["ctx"] = Clusterer(w, h, case["dt"], max_disorder=t)
        state["start"] = state["ctx"].snapshot()
    else:
        state["hits"] = hits.cpu().numpy().view(HIT_DTYPE).reshape(-1)
        state["records"] = np.zeros(n, dtype=CLUSTER_DTYPE)
        state["ctx"] = Clusterer(w, h, case["dt"], case["variant"])
    torch.cuda.synchronize()
    return state


# ---------------------------------------------------------------------------
# one pass


def _outputs(labels, records):
    """Labels, the records' whole-number fields and their centroids (views)."""
    return {"labels": labels, "whole": records.view(torch.int64)[:, :4],
            "centroid": records.view(torch.float32)[:, 8:10]}


def _acquisition(state):
    """A whole acquisition: chunks in, what each finalises out."""
    ctx, hits, n, step = state["ctx"], state["hits"], state["case"]["n"], state["case"]["parts"]
    labels, indices, records = state["labels"], state["indices"], state["records"]
    ctx.restore(state["start"])
    done, found, ends = 0, 0, []
    for a in list(range(0, n, step)) + [n]:
        if a < n:
            ctx.push_ptr(hits[a].data_ptr(), min(step, n - a), False)
        else:
            ctx.flush()
        done += ctx.labels_into(labels.data_ptr() + 8 * done, n - done, False, indices.data_ptr() + 8 * done)
        found += ctx.features_into(records.data_ptr() + 40 * found, n - found, False)
        ends.append((done, found))
    return dict(_outputs(labels, records), indices=indices, ends=np.array(ends, dtype=np.int64))


def run(state):
    call = state["call"]
    if call == "fixed":
        c, hits, labels, records = state["case"], state["hits"], state["labels"], state["records"]
        status = state["lib"].tpc_cluster_static(
            hits.data_ptr(), c["n"], c["width"], c["height"], c["dt"], labels.data_ptr(), records.data_ptr(),
            c["n"], state["counts"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        if status:
            raise RuntimeError("tpc_cluster_static: status %d" % status)
        return dict(_outputs(labels, records), counts=state["counts"])
    if call == "batch":
        for d in state["dets"]:
            d["ctx"].push_ptr(d["hits"].data_ptr(), d["hits"].shape[0], True)
        batch_flush([d["ctx"] for d in state["dets"]])
        counts = np.array([d["ctx"].counts() for d in state["dets"]], dtype=np.int64)
        return {"detectors": [_outputs(d["labels"], d["records"]) for d in state["dets"]], "counts": counts}
    if call == "stream":
        return _acquisition(state)
    ctx = state["ctx"]
    if call == "bound":
        ctx.push_ptr(state["hits"].data_ptr(), state["hits"].shape[0], True)
        ctx.flush()
        return dict(_outputs(state["labels"], state["records"]), clusters=ctx.counts()[1])
    ctx.push(state["hits"])
    ctx.flush()
    records = state["records"]
    if call == "oneshot":
        labels = ctx.labels(device=True)
        found = ctx.features_into(records.data_ptr(), records.shape[0], True)
        return dict(_outputs(labels, records), clusters=found)
    labels = ctx.labels()
    found = ctx.features_into(records.ctypes.data, records.shape[0], False)
    return dict(_outputs(torch.from_numpy(labels.view(np.int64)), torch.from_numpy(records.view(np.uint8).reshape(-1, 40))),
                clusters=found)


def work(case):
    """Every hit read once (16 B), every label (8 B; its index too when
    streaming) and every cluster record (40 B) written once; the sums of the
    centroid are four operations a hit."""
    per_cluster = {"global": 1000.0, "static": 9.5}.get(case["variant"], 19.0) if case["mix"] else 3.3
    per_hit = 16 + (16 if case["call"] == "stream" else 8) + 40 / per_cluster
    return {"bytes": case["n"] * per_hit, "flops": 4.0 * case["n"]}


# ---------------------------------------------------------------------------
# the centroids in 64 bits


def _components(pix, toa, width, height, dt):
    """Smallest hit index of each hit's cluster.  A hit is joined to the latest
    hit at or before it on each of its nine pixels if that one lies within dt:
    earlier ones within dt are joined to that one along their own pixel."""
    n, dev = pix.numel(), pix.device
    t = toa - toa.min()
    key, order = torch.sort((pix << 40) | t, stable=True)
    label = torch.arange(n, device=dev)
    x, y = pix % width, pix // width
    heads, tails = [], []
    same = (key[1:] >> 40 == key[:-1] >> 40) & (key[1:] - key[:-1] <= dt)
    heads.append(order[1:][same])
    tails.append(order[:-1][same])
    for dy in (-1, 0, 1):
        for dx in (-1, 0, 1):
            if dx == 0 and dy == 0:
                continue
            inside = (x + dx >= 0) & (x + dx < width) & (y + dy >= 0) & (y + dy < height)
            want = ((y + dy) * width + x + dx) << 40 | t
            at = torch.searchsorted(key, want, right=True) - 1
            found = key[at.clamp(min=0)]
            ok = inside & (at >= 0) & (found >> 40 == want >> 40) & (want - found <= dt)
            heads.append(torch.nonzero(ok).view(-1))
            tails.append(order[at[ok]])
    a, b = torch.cat(heads), torch.cat(tails)
    while a.numel():
        la, lb = label[a], label[b]
        apart = la != lb
        a, b, la, lb = a[apart], b[apart], la[apart], lb[apart]
        label.scatter_reduce_(0, torch.maximum(la, lb), torch.minimum(la, lb), "amin")
        while True:
            up = label[label]
            if torch.equal(up, label):
                break
            label = up
    return label


def _centroids(case, hits, width, height, marks=None):
    """Centroids of the clusters in label order, zeros behind the last one.  A
    stream's come in the order of their steps: a cluster is final at the first
    step whose watermark (``marks``) its last ToA does not exceed."""
    x, y, tot, toa = hits[:, 0] & 0xFFFF, (hits[:, 0] >> 16) & 0xFFFF, (hits[:, 0] >> 32) & 0xFFFF, hits[:, 1]
    n, dev = toa.numel(), toa.device
    label = _components(y * width + x, toa, width, height, case["dt"])
    root = label == torch.arange(n, device=dev)
    k = (torch.cumsum(root, 0) - 1)[label]
    m = int(root.sum())

    def total(v):
        return torch.zeros(m, dtype=torch.int64, device=dev).scatter_add_(0, k, v)

    weight = total(tot).to(torch.float64)
    c = torch.stack([total(tot * x) / weight, total(tot * y) / weight], 1)
    if marks is not None:
        last = torch.zeros(m, dtype=torch.int64, device=dev).scatter_reduce_(0, k, toa, "amax")
        step = torch.searchsorted(torch.tensor(marks, dtype=torch.int64, device=dev), last)
        c = c[torch.sort(step, stable=True).indices]
    return torch.cat([c, torch.zeros((n - m, 2), dtype=torch.float64, device=dev)])


def exact(case, seed):
    if case["variant"] != "local":
        return None
    none = {"labels": None, "whole": None}
    if case["call"] == "batch":
        found = []
        for i, (dw, dh, dn, rate) in enumerate(_detectors(case)):
            hits, _ = _stream(case, dn, dw, dh, rate, seed * 64 + i)
            found.append(dict(none, centroid=_centroids(case, hits, dw, dh)))
        return {"detectors": found, "counts": None}
    w, h, n = case["width"], case["height"], case["n"]
    hits, t = _stream(case, n, w, h, case["rate"], seed)
    if case["call"] == "stream":
        seen = _prefix_max(hits[:, 1])
        marks = [int(seen[min(a + case["parts"], n) - 1]) - t - case["dt"] for a in range(0, n, case["parts"])]
        return dict(none, centroid=_centroids(case, hits, w, h, marks), indices=None, ends=None)
    c = _centroids(case, hits, w, h)
    return dict(none, centroid=c, **({"counts": None} if case["call"] == "fixed" else {"clusters": None}))
