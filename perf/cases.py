"""The work that programs built on this library have it do, as cases that can be timed.

Each case is one pass through public entry points, on seeded synthetic events of
``paper_1310_7556_gb300.eventgen``: single events from the smallest grid to the finest one, host
hits end to end, every accumulator and axis option, batches and the server.  ``listed()`` gives the
standing cases, ``draw(rng)`` others of the same ranges, ``prepare`` what a program holds before the
call, ``run`` the pass and its outputs, ``work`` the bytes and operations no implementation can do
without, ``exact`` the outputs in 64 bits where they have a value of their own.

Candidate lists are whole numbers (cells, layer masks, counts of hits), decided cell by cell: they
are the same or they are wrong, and have no 64-bit value to be near to.  The accumulator of a vote
has one, cell by cell.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1310_7556_gb300 import binding
from paper_1310_7556_gb300 import eventgen as eg

# ---------------------------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------------------------

# Fields of every case: path (which entry points), layers ("barrel": the ten uneven layers of the
# synthetic detector, "paper": ten even ones, or a number of even layers out to 110 cm), the grid
# (n_qpt rows over +-qpt, n_phi columns, n_d0 slices over +-d0 cm), counts (vote counts instead of
# layer masks), the peak threshold, the tracks and noise hits of the event, their pT range, the
# radius jitter (cm); for several events at once: events, tracks then being the most per event.
_DEFAULTS = dict(path="event", layers="barrel", n_qpt=512, n_phi=2048, qpt=2.0, n_d0=0, d0=0.0, counts=False,
                 threshold=7, tracks=5000, noise=50000, pt_lo=0.5, pt_hi=100.0, jitter=0.0, events=1)


def _case(**kw):
    return {**_DEFAULTS, **kw}


def listed():
    return [
        # a quiet event on a coarse grid, hits already on the GPU: what a call costs at all
        _case(name="single_50trk", n_qpt=128, n_phi=256, qpt=1.0, threshold=8, tracks=50, noise=0, pt_lo=1.0, pt_hi=50.0),
        # a high-pileup event (100k hits), hits on the GPU: the plain method's standing workload
        _case(name="pileup_event"),
        # the same event from pinned host memory, candidates back on the host: a trigger's whole call
        _case(name="pileup_host", path="host"),
        # fine binning: 420k hits on four million cells
        _case(name="fine_event", n_qpt=1024, n_phi=4096, tracks=20000, noise=200000),
        # the paper's own detector and 2048 x 2048 grid; many candidates of a busy event to confirm
        _case(name="paper_2000trk", layers="paper", n_qpt=2048, n_phi=2048, qpt=1.0, threshold=8, tracks=2000, noise=0,
              pt_lo=1.0),
        # a detector whose modules lie within +-0.5 cm of their layer's radius: each hit its own radius
        _case(name="jittered_event", jitter=0.5),
        # the paper's literal accumulator, A[B[i]] += 1
        _case(name="counts_event", counts=True, threshold=70),
        # non-prompt tracks: a third axis of impact parameters
        _case(name="displaced_event", n_qpt=256, qpt=1.0, n_d0=16, d0=2.0, threshold=8, tracks=200, noise=1000, pt_lo=2.0),
        # the vote alone into a caller's accumulator, for programs that may not allocate
        _case(name="vote_static", path="static"),
        # a few events per launch, as a latency-bound trigger collects them
        _case(name="batch_16", path="batch", events=16, tracks=10000),
        # many events per launch: offline reprocessing, the throughput path
        _case(name="batch_256", path="batch", events=256, tracks=10000),
        # a burst of events through the continuous-batching server, host to host
        _case(name="served_24", path="served", events=24, tracks=10000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["event", "event", "host", "fine", "paper", "jittered", "counts", "displaced", "static", "batch",
                       "batch", "served"])
    if kind in ("batch", "served"):
        events = _log_int(rng, 2, 160) if kind == "batch" else rng.randint(4, 32)
        return _case(path=kind, events=events, n_qpt=_log_int(rng, 128, 512), n_phi=64 * rng.randint(8, 32),
                     tracks=_log_int(rng, 1000, 10000), threshold=rng.choice([7, 8]))
    if kind == "paper":
        return _case(layers="paper", n_qpt=_log_int(rng, 512, 2048), n_phi=64 * rng.randint(16, 32), qpt=1.0, threshold=8,
                     tracks=_log_int(rng, 10, 2500), noise=0, pt_lo=1.0)
    if kind == "displaced":
        counts = rng.random() < 0.3
        return _case(n_qpt=_log_int(rng, 64, 256), n_phi=64 * rng.randint(8, 32), qpt=1.0, n_d0=rng.randint(3, 16),
                     d0=rng.choice([1.0, 2.0]), counts=counts, threshold=8, tracks=_log_int(rng, 20, 400),
                     noise=_log_int(rng, 10, 2000), pt_lo=2.0)
    # prompt events: small to pileup sizes, 6 to 12 layers, grids with odd numbers of rows
    layers = rng.choice(["barrel", "barrel", "barrel", 6, 12])
    n_layers = 10 if layers == "barrel" else layers
    n_qpt, n_phi = _log_int(rng, 65, 700), 64 * rng.randint(4, 40)
    tracks = _log_int(rng, 10, 6000)
    if kind == "fine":
        n_qpt, n_phi, tracks = _log_int(rng, 600, 1024), 64 * rng.randint(40, 64), _log_int(rng, 500, 20000)
    noise = int(tracks * n_layers * rng.uniform(0.0, 1.0))
    case = _case(layers=layers, n_qpt=n_qpt, n_phi=n_phi, qpt=rng.choice([1.0, 2.0]), threshold=max(3, n_layers - 3),
                 tracks=tracks, noise=noise)
    if kind == "host":
        case["path"] = "host"
    elif kind == "static":
        # the call's limits: 131,072 hits, 1,024 rows, 4,096 columns
        case.update(path="static", tracks=min(tracks, 5000), counts=rng.random() < 0.3)
        case["noise"] = min(noise, 50000)
    elif kind == "jittered":
        case["jitter"] = rng.choice([0.1, 0.5])
    elif kind == "counts":
        # a threshold near the top of the event's own occupancy
        mean = (tracks * n_layers + noise) / n_phi
        case.update(counts=True, threshold=max(n_layers - 2, int(mean + 3.0 * math.sqrt(mean))))
    return case


# ---------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------

def _workload(case):
    layers = case["layers"]
    if layers == "barrel":
        geometry = eg.Geometry()
    elif layers == "paper":
        geometry = eg.PAPER_GEOMETRY
    else:
        geometry = eg.Geometry(radii_cm=tuple(110.0 * k / layers for k in range(1, layers + 1)))
    b = eg.Binning(n_qpt=case["n_qpt"], qpt_min=-case["qpt"], qpt_max=case["qpt"], n_phi=case["n_phi"],
                   threshold=case["threshold"], accumulator=eg.ACC_COUNTS if case["counts"] else eg.ACC_LAYERS,
                   n_d0=case["n_d0"], d0_min=-case["d0"] if case["n_d0"] else -1.0,
                   d0_max=case["d0"] if case["n_d0"] else 1.0)
    common = dict(binning=b, geometry=geometry, pt_range=(case["pt_lo"], case["pt_hi"]), radius_jitter_cm=case["jitter"],
                  d0_range=(-case["d0"], case["d0"]) if case["n_d0"] else ())
    if layers == "paper":   # the paper's simulation is of the transverse plane, 0.4 mm resolution
        common.update(smear_rphi_cm=0.04, eta_max=0.0, z0_sigma_cm=0.0)
    if case["events"] > 1:
        return eg.Workload("events", tracks_log_uniform=(min(100, case["tracks"]), case["tracks"]),
                           noise_fraction=(0.5, 2.0), **common)
    return eg.Workload("event", n_tracks=case["tracks"], n_noise=case["noise"], **common)


_FIELDS = ("r", "phi", "z", "layer")


def _cells(case):
    return case["n_qpt"] * max(1, case["n_d0"]) * case["n_phi"]


class _State:
    pass


def _records(n):
    """Room for n candidate records on the GPU; what a pass does not fill stays zero."""
    return torch.zeros((n, 8), dtype=torch.int32, device="cuda")


def prepare(case, seed):
    w = _workload(case)
    s = _State()
    s.path, s.w = case["path"], w
    s.stream = torch.cuda.current_stream()
    if case["events"] > 1:
        events = [w.event(i, base_seed=seed) for i in range(case["events"])]
    else:
        events = [w.event(0, base_seed=seed)]
    most = max(e.n_hits for e in events)
    # no two candidates touch, so a grid holds at most a quarter of its cells of them
    cap = max(1, _cells(case) // 4)
    if s.path in ("event", "host"):
        s.n = most
        s.ctx = binding.HoughContext(w.geometry, w.binning, max_hits=max(most, 1), max_candidates=cap, max_members=1 << 24)
        s.cap = cap
    if s.path == "host":
        s.hits = [torch.from_numpy(getattr(events[0], k)).pin_memory() for k in _FIELDS]
        s.out = np.zeros(cap, dtype=binding.CANDIDATE_DTYPE)
    elif s.path == "served":
        s.events = events
        s.server = binding.HoughServer(w.geometry, w.binning, max_batch_events=16, max_batch_hits=16 * most, lanes=4,
                                       max_in_flight=3, max_candidates=min(cap, 1 << 17))
        s.out = np.zeros((len(events), min(cap, 1 << 17)), dtype=binding.CANDIDATE_DTYPE)
        s.found = np.zeros(len(events), dtype=np.int64)
    else:
        s.hits = [torch.from_numpy(np.concatenate([getattr(e, k) for e in events])).cuda() for k in _FIELDS]
        if s.path == "event":
            s.out = _records(cap)
        elif s.path == "static":
            s.n = most
            s.cells = torch.empty((case["n_qpt"], case["n_phi"]), dtype=torch.int16, device="cuda")
        else:
            s.start = np.zeros(len(events) + 1, dtype=np.int64)
            s.start[1:] = np.cumsum([e.n_hits for e in events])
            s.batch = binding.HoughBatch(w.geometry, w.binning, max_events=len(events), max_hits=int(s.start[-1]),
                                         max_candidates=min(cap, 1 << 17))
            s.cap = len(events) * min(cap, 1 << 16)
            s.out = _records(s.cap)
            s.offsets = np.zeros(len(events) + 1, dtype=np.int64)
    return s


# ---------------------------------------------------------------------------------------------
# The pass
# ---------------------------------------------------------------------------------------------

def _ok(rc):
    if rc != binding.OK:
        raise binding.HoughError(rc, binding.load().hough_last_error().decode())


def _words(records):
    return records.view(np.uint32).view(np.int32)


def run(s):
    lib = binding.load()
    stream = s.stream.cuda_stream
    if s.path == "event":
        # the whole path on device-resident hits, candidates left on the device
        n = ctypes.c_int32(0)
        r, phi, z, layer = (t.data_ptr() for t in s.hits)
        _ok(lib.hough_process(s.ctx._h, r, phi, z, layer, s.n, s.out.data_ptr(), s.cap, ctypes.byref(n), binding.DEVICE,
                              stream))
        return [s.out, n.value]
    if s.path == "host":
        got = s.ctx.process(*s.hits, n_hits=s.n, cap=s.cap, out=s.out, stream=stream)
        return [_words(s.out), got.shape[0]]
    if s.path == "static":
        binding.vote_static(s.w.geometry, s.w.binning, *s.hits, s.n, s.cells, stream=stream)
        return s.cells
    if s.path == "batch":
        s.batch.run(*s.hits, s.start, where=binding.DEVICE, stream=stream)
        _ok(lib.hough_batch_candidates(s.batch._h, s.out.data_ptr(), s.cap, s.offsets.ctypes.data, binding.DEVICE, stream))
        return [s.out, s.offsets]
    # served: a burst submitted as it comes, results taken in order; a refused event waits for the oldest
    waiting, nxt, done = [], 0, 0
    result = binding.ServeResult()
    while done < len(s.events):
        if nxt < len(s.events):
            ticket = s.server.submit_event(s.events[nxt])
            if ticket is not None:
                waiting.append(ticket)
                nxt += 1
                continue
        _ok(lib.hough_serve_poll(s.server._h, waiting.pop(0), s.out[done].ctypes.data, s.out.shape[1], ctypes.byref(result),
                                 10_000_000))
        s.found[done] = result.n_candidates
        done += 1
    return [_words(s.out), s.found]


def work(case):
    """Hits read once (13 bytes each), the cells of a bare vote written once or a record per track (32
    bytes); a comparison and an OR or addition for each vote, or, where fewer, each (cell, layer)."""
    layers = 10 if case["layers"] in ("barrel", "paper") else case["layers"]
    rows = case["n_qpt"] * max(1, case["n_d0"])
    tracks, hits = case["tracks"], case["tracks"] * layers + case["noise"]
    if case["events"] > 1:   # log-uniform tracks per event, noise 0.5 to 2 times their hits
        lo = min(100, tracks)
        tracks = case["events"] * ((tracks - lo) / math.log(tracks / lo) if tracks > lo else tracks)
        hits = tracks * layers * 2.25
    out = 2 * _cells(case) if case["path"] == "static" else 32 * tracks
    decisions = min(hits * rows, case["events"] * _cells(case) * layers) if not case["counts"] else hits * rows
    return {"bytes": 13 * hits + out, "flops": 2 * decisions}


def exact(case, seed):
    """The accumulator of a bare vote, evaluated as the method defines it: hit by hit, row by row."""
    if case["path"] != "static":
        return None
    w = _workload(case)
    e, b, g = w.event(0, base_seed=seed), w.binning, w.geometry
    r, phi = e.r.astype(np.float64), e.phi.astype(np.float64)
    cells = np.zeros((b.n_qpt, b.n_phi), dtype=np.int64)
    dk = (b.qpt_max - b.qpt_min) / b.n_qpt
    coef = 0.15 * g.b_tesla * (r / 100.0)
    by_layer = [np.flatnonzero(e.layer == l) for l in range(g.n_layers)]
    for i in range(b.n_qpt):
        x = coef * (b.qpt_min + (i + 0.5) * dk)
        fits = np.abs(x) <= 1.0
        phi0 = phi - np.arcsin(np.where(fits, x, 0.0))
        j = np.mod(np.floor(b.n_phi * (phi0 + math.pi) / (2.0 * math.pi)).astype(np.int64), b.n_phi)
        if case["counts"]:
            cells[i] = np.minimum(np.bincount(j[fits], minlength=b.n_phi), 65535)
        else:
            for l, hits in enumerate(by_layer):
                cells[i, j[hits[fits[hits]]]] |= 1 << l
    return cells.astype(np.uint16).view(np.int16)
