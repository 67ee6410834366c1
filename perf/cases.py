"""What a user of the track finder has it do, as cases that can be timed.

A case is a dict of plain values.  ``prepare`` makes what a program has in
hand before the call (hits, and the context, batch, sectors or server object
that it keeps), ``run`` makes one pass through the public entry points and
returns everything that the pass produces, and ``work`` states the bytes and
operations that the pass cannot do without.

Every output is a whole number: vote counts, peak totals, and 32-byte peak
records, whose two cell centres are compared by their bits.  The records that
a pass does not write stay zero.
"""
import numpy as np
import torch

from paper_1507_03074_gb300 import ht, synth

PEAK_WORDS = 8      # int32 words of one peak record
CAPACITY = 1 << 16  # peaks a caller makes room for
REQUEST_CAPACITY = 1 << 12  # and for one request to the server

_DEFAULTS = dict(kind="event", n_theta=4, n_phi=16, n_a=1024, n_b=1024, win=0, threshold=10, hits=4990,
                 events=1, parts=1, sectors=1, peaks_only=False, four_d=False, matrix=False)


def _case(name=None, **kw):
    c = dict(_DEFAULTS, **kw)
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # the smallest call: ten tracks in 8 slices of 64 x 64 cells, as a trigger primitive or a unit test of a
        # user's program runs it; launches and latency are all there is.  The matrix is handed on.
        _case("tiny_event", n_theta=2, n_phi=4, n_a=64, n_b=64, threshold=8, hits=120, matrix=True),
        # the paper's event, hits on the device, the call that the project is about
        _case("paper_event"),
        # the same event from host arrays to a host peak list, one blocking round trip: the latency of one event
        _case("paper_host", kind="host"),
        # the same event when only the peak list is wanted
        _case("paper_peaks_only", peaks_only=True),
        # admission windows of one bin in theta and phi, so that a track which crosses a slice edge keeps all its
        # votes: nine times the votes, thousands of candidates
        _case("paper_windows", win=1),
        # the paper's event arriving in four read-out fragments that are added up, then searched, and the matrix
        # handed to the caller's own analysis
        _case("paper_fragments", kind="parts", parts=4, matrix=True),
        # the paper's four phi sectors, merged into one peak list
        _case("paper_sectors", kind="sectors", sectors=4),
        # odd bin counts (rows that are not 16-byte multiples, slices that start anywhere), and the 80-neighbour
        # peak rule
        _case("odd_bins_4d", n_a=999, n_b=1001, four_d=True),
        # the upgrade event: 50 000 hits in a 4 GiB matrix
        _case("upgrade_event", n_theta=8, n_phi=32, n_a=2048, n_b=2048, hits=50000),
        # a hundred uneven events from page-locked host memory in one batch: the largest call
        _case("batch_uneven", kind="batch", events=100, hits=5000),
        # the maxima step alone on two matrices that the caller holds, for programs that may not allocate
        _case("scan_held", kind="scan", events=2),
        # a burst of requests of uneven size and two binnings to the server
        _case("serve_burst", kind="serve", events=24, hits=3000),
    ]


def _between(rng, lo, hi):
    """A whole number in [lo, hi], even over its logarithm."""
    return min(hi, max(lo, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    kind = rng.choice(["event", "event", "event", "host", "parts", "sectors", "batch", "scan", "serve"])
    n_theta, n_phi = _between(rng, 1, 8), _between(rng, 2, 32)
    n_a, n_b = _between(rng, 48, 2048), _between(rng, 48, 2048)
    if rng.random() < 0.5:
        n_b = max(48, n_b // 4 * 4)
    while n_theta * n_phi * n_a * n_b > (1 << 30 if kind == "event" else 1 << 28):
        n_a = max(48, n_a // 2)
    c = dict(kind=kind, n_theta=n_theta, n_phi=n_phi, n_a=n_a, n_b=n_b, threshold=rng.choice([8, 9, 10, 11, 12]))
    c["matrix"] = kind in ("event", "parts") and rng.random() < 0.25
    if kind == "event":
        c["peaks_only"] = not c["matrix"] and rng.random() < 0.3
        c["win"] = 1 if n_theta > 2 and n_phi > 4 and rng.random() < 0.3 else 0
        c["four_d"] = not c["peaks_only"] and rng.random() < 0.3
    # occupancy: from nearly empty slices to a quarter of a hit per column
    most = max(60, int(0.25 * n_theta * n_phi * n_b / (9 if c.get("win") else 1)))
    c["hits"] = min(50000, _between(rng, 50, most))
    if kind == "parts":
        c["parts"] = rng.randint(2, 6)
    if kind == "sectors":
        c["sectors"] = rng.choice([s for s in range(1, 9) if n_phi % s == 0])
    if kind in ("batch", "scan", "serve"):
        cells = n_theta * n_phi * n_a * n_b
        c["events"] = _between(rng, 2, max(2, min(64, (1 << 31) // cells if kind == "batch" else (1 << 29) // cells)))
        c["peaks_only"] = kind == "batch" and rng.random() < 0.4
        c["hits"] = max(50, min(c["hits"], 5000))
    return _case(**c)


def _binning(c):
    return ht.Binning(c["n_theta"], c["n_phi"], c["n_a"], c["n_b"], c["win"], c["win"])


def _hits(n, seed):
    """One synthetic event of n hits: helices on 12 layers and some noise, as float32 arrays."""
    ev = synth.make_event(*synth.split_hits(n), seed=seed)
    return ev.x, ev.y, ev.z


def _uneven(c, seed):
    """The events of a batch, burst or scan: a tenth of c["hits"] to all of it, each of its own size (the same sizes
    for every seed)."""
    rng = np.random.default_rng(1000)
    return [_hits(int(n), seed * 128 + i)
            for i, n in enumerate(rng.integers(max(c["hits"] // 10, 12), c["hits"] + 1, c["events"]))]


def _pinned(a):
    """A page-locked copy of a host array, as a numpy array."""
    return torch.from_numpy(np.ascontiguousarray(a)).pin_memory().numpy()


def _device(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _records(n):
    return torch.zeros(n, PEAK_WORDS, dtype=torch.int32, device="cuda")


def _keep(rows, peaks):
    """A host peak list into the caller's own rows."""
    rows[:len(peaks)] = peaks.view(np.int32).reshape(-1, PEAK_WORDS)
    return rows


def prepare(case, seed):
    c = dict(_DEFAULTS, **case)
    b, r, T, kind = _binning(c), ht.Ranges(), c["threshold"], c["kind"]
    s = {"case": c, "binning": b, "ranges": r}
    if kind in ("event", "parts"):
        x, y, z = (_device(a) for a in _hits(c["hits"], seed))
        cut = [i * c["hits"] // c["parts"] for i in range(c["parts"] + 1)]
        s["hits"] = [(x[i:j].clone(), y[i:j].clone(), z[i:j].clone()) for i, j in zip(cut, cut[1:])]
        s["obj"] = ht.Context(b, r, threshold=T, max_hits=c["hits"])
        if c["matrix"]:
            s["M"] = torch.zeros(b.shape(), dtype=torch.int32, device="cuda")
    elif kind == "host":
        s["hits"] = _hits(c["hits"], seed)
        s["obj"] = ht.Context(b, r, threshold=T, max_hits=c["hits"])
    elif kind == "sectors":
        s["hits"] = tuple(_device(a) for a in _hits(c["hits"], seed))
        s["obj"] = ht.Sectors(b, r, threshold=T, n_sectors=c["sectors"], max_hits=c["hits"])
    elif kind == "batch":
        x, y, z, off = ht.Batch.concat(_uneven(c, seed))
        s["hits"] = (_pinned(x), _pinned(y), _pinned(z), off)
        s["obj"] = ht.Batch(b, r, threshold=T, max_events=c["events"], max_hits=int(off[-1]), capacity=CAPACITY)
    elif kind == "scan":
        s["M"] = torch.empty((c["events"],) + b.shape(), dtype=torch.int32, device="cuda")
        with ht.Context(b, r, threshold=T, max_hits=c["hits"]) as ctx:
            for e, hits in enumerate(_uneven(c, seed)):
                ctx.fill(*(_device(a) for a in hits))
                ctx.matrix_into(s["M"][e])
                ctx.sync()
    elif kind == "serve":
        # nine requests of ten in the case's binning, the tenth in one of half the bins in A and B
        half = ht.Binning(b.n_theta, b.n_phi, max(b.n_a // 2, 1), max(b.n_b // 2, 1))
        s["requests"] = [(half if i % 10 == 9 else b, r, T) + h for i, h in enumerate(_uneven(c, seed))]
        s["rows"] = [np.zeros((REQUEST_CAPACITY, PEAK_WORDS), np.int32) for _ in s["requests"]]
        s["obj"] = ht.Server(hbm_budget_bytes=16 << 30, max_batch=8, max_hits_per_event=c["hits"])
        _serve(s)  # a server that is up has its lanes
    if kind in ("host", "batch"):
        s["rows"] = np.zeros((CAPACITY, PEAK_WORDS), np.int32)
    elif kind in ("event", "parts", "sectors"):
        s["out"], s["count"] = _records(CAPACITY), torch.zeros(1, dtype=torch.int32, device="cuda")
    elif kind == "scan":
        per = CAPACITY // c["events"]
        s["out"], s["count"] = _records(per * c["events"]), torch.zeros(c["events"], dtype=torch.int32, device="cuda")
    return s


def _serve(s):
    tickets = [s["obj"].submit(*q) for q in s["requests"]]
    peaks, totals = [], []
    for t, rows in zip(tickets, s["rows"]):
        got = None
        while got is None:
            got = s["obj"].poll(t, capacity=REQUEST_CAPACITY, timeout_us=1000000)
        peaks.append(_keep(rows, got[1]))
        totals.append(got[2])
    return {"peaks": peaks, "totals": np.array(totals, np.int64)}


def run(state):
    s = state
    c, kind = s["case"], s["case"]["kind"]
    if kind in ("event", "parts"):
        ctx = s["obj"]
        for i, (x, y, z) in enumerate(s["hits"]):
            ctx.fill(x, y, z, accumulate=i > 0, peaks_only=c["peaks_only"])
        ctx.find_maxima(capacity=CAPACITY, out=s["out"], count=s["count"], four_d=c["four_d"])
        got = {"peaks": s["out"], "total": s["count"]}
        if c["matrix"]:
            ctx.matrix_into(s["M"])
            got["matrix"] = s["M"]
        return got
    if kind == "host":
        s["obj"].fill(*s["hits"], peaks_only=c["peaks_only"])
        peaks, total = s["obj"].find_maxima(capacity=CAPACITY)
        return {"peaks": _keep(s["rows"], peaks), "total": total}
    if kind == "sectors":
        s["obj"].fill(*s["hits"])
        s["obj"].find_maxima(capacity=CAPACITY, out=s["out"], count=s["count"])
        return {"peaks": s["out"], "total": s["count"]}
    if kind == "batch":
        peaks, counts = s["obj"].run(*s["hits"], peaks_only=c["peaks_only"])
        return {"peaks": _keep(s["rows"], peaks), "counts": counts}
    if kind == "scan":
        ht.find_maxima_noalloc(s["binning"], s["ranges"], c["threshold"], s["M"], c["events"], s["out"],
                               CAPACITY // c["events"], s["count"])
        return {"peaks": s["out"], "counts": s["count"]}
    return _serve(s)


def work(case):
    """Hits read once and the matrix written once (read once by the scan alone; read and written once more where it
    is handed on; not touched where only peaks are wanted); six operations for the B bin of every (hit, admitted
    slice, A bin), one comparison per cell that the scan alone reads."""
    c = dict(_DEFAULTS, **case)
    cells = c["n_theta"] * c["n_phi"] * c["n_a"] * c["n_b"]
    if c["kind"] == "scan":
        return {"bytes": 4.0 * cells * c["events"], "flops": 1.0 * cells * c["events"]}
    n = c["hits"]
    if c["kind"] in ("batch", "serve"):
        n = 0.55 * c["hits"] * c["events"]
        cells *= c["events"] if c["kind"] == "batch" else c["events"] - 0.75 * (c["events"] // 10)
    w = c["win"]
    slices = (2 * w + 1 - w * (w + 1) / c["n_theta"]) * min(2 * w + 1, c["n_phi"])
    moved = 0 if c["peaks_only"] else 12.0 * cells if c["matrix"] else 4.0 * cells
    return {"bytes": 12.0 * n + moved, "flops": 6.0 * n * slices * c["n_a"]}


def exact(case, seed):
    """None: no output is a computed real number.  A vote goes to the bin that the stated binary32 rule names, so 64
    bits would count other votes, and totals, indices and records are compared as whole numbers."""
    return None
