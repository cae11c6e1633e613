"""The work that users of the track-finding library have it do, as cases that
can be timed: ``listed()`` names them, ``draw(rng)`` gives more of the same
ranges, ``prepare(case, seed)`` makes what a program has in hand before the
call, ``run(state)`` is one pass through the public entry points.

Every output of the library is a whole number defined bit for bit by its
header, so two correct programs give equal outputs.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2511_02742_gb300 import hough, synth

POOL_TRACKS = 2048          # generated helices per seed; windows draw from them
STEP_PS, OVERLAP = 5000, 2  # 10 ns windows sliding by 5 ns
EXT_TOL = 16 * 38           # track extension tolerance: 16 strips
MAX_TRACKS = 64             # lines the iterative search may take per window
MAX_PEAKS = 64              # the library's default
# mean hits of a track: one turn at 100-300 MeV/c, four turns at 50-300
HITS_PER_TRACK = {1: 14.0, 4: 22.8}


def listed():
    pileup = dict(law="poisson", tracks=10, noise=0.02, turns=1, encoded=False)
    return [
        # an event display or a trigger loop that looks at single windows as
        # they come: latency of one call
        dict(name="one_window", kind="find", n_theta=512, n_rho=512, windows=1, **pileup),
        # an ordinary small job: 1000 windows of 5 tracks
        dict(name="plain_1000", kind="find", n_theta=512, n_rho=512, windows=1000, law="fixed",
             tracks=5, noise=0.01, turns=1, encoded=False),
        # offline processing: a large uneven batch replayed from a graph
        dict(name="batched_1e5", kind="plan", n_theta=512, n_rho=512, windows=100000, **pileup),
        # a batch with a long tail of heavy windows, hits already encoded
        dict(name="uneven_heavy", kind="find", n_theta=512, n_rho=512, windows=4000,
             law="uniform", tracks=40, noise=0.02, turns=1, encoded=True),
        # the highest pileup, about 1000 hits a window
        dict(name="high_pileup_1e4", kind="find", n_theta=1024, n_rho=1024, windows=10000,
             law="fixed", tracks=40, noise=0.05, turns=4, encoded=False),
        # the paper's own binning, neither side a power of two
        dict(name="paper_180x1000", kind="find", n_theta=180, n_rho=1000, windows=3001, **pileup),
        # the find with every accumulator kept, for study of the peak rule
        dict(name="export_high_pileup", kind="export", n_theta=1024, n_rho=1024, windows=500,
             law="fixed", tracks=40, noise=0.05, turns=4, encoded=False),
        # accumulators alone, for a program with a peak finder of its own
        dict(name="accumulate_high_pileup", kind="accumulate", n_theta=1024, n_rho=1024,
             windows=500, law="fixed", tracks=40, noise=0.05, turns=4, encoded=False),
        # online serving: one time slice from host memory to host memory
        dict(name="serve_slice", kind="serve", n_theta=512, n_rho=512, windows=100,
             law="uniform", tracks=40, noise=0.02, turns=1, encoded=False),
        # the highest bin taken and removed until no line is left
        dict(name="iterative_5000", kind="iterative", n_theta=512, n_rho=512, windows=5000,
             **pileup),
        # the paper's two-stage search, one line a window
        dict(name="coarse_fine_1e5", kind="coarse_fine", n_theta=512, n_rho=512, windows=100000,
             **pileup),
        # a whole readout: 200 us of detector time cut into overlapping
        # windows, searched, the tracks extended
        dict(name="stream_200us", kind="stream", n_theta=512, n_rho=512, windows=40001,
             law="rate", tracks=0.6, noise=0.02, turns=1, encoded=False),
    ]


def _log(rng, lo, hi):
    return lo * math.exp(rng.random() * math.log(hi / lo))


def draw(rng):
    kind = rng.choice(["find"] * 5 + ["plan", "export", "accumulate", "serve", "iterative",
                                      "coarse_fine", "stream"])
    shape = rng.choice([(256, 256), (512, 512), (512, 512), (180, 1000), (1024, 1024), None])
    if shape is None:
        shape = (int(_log(rng, 100, 1024)), 4 * int(_log(rng, 50, 256)))
    turns = 4 if min(shape) >= 1000 and rng.random() < 0.5 else 1
    law = rng.choice(["fixed", "poisson", "uniform"])
    tracks = max(1, int(_log(rng, 1, 41)))
    if kind == "stream":
        law, tracks, turns = "rate", round(_log(rng, 0.06, 1.5), 3), 1
    case = dict(kind=kind, n_theta=shape[0], n_rho=shape[1], windows=1, law=law, tracks=tracks,
                noise=rng.choice([0.0, 0.01, 0.02, 0.05]), turns=turns,
                encoded=rng.random() < 0.4)
    # as many windows as keep a pass below the largest listed ones
    hits = _hits_per_window(case)
    if kind in ("export", "accumulate"):
        most = min(5000, 2e9 / (4 * shape[0] * shape[1]))
    elif kind == "iterative":
        most = min(5000, 3.5e9 / (hits * shape[0] * _mean_tracks(case)))
    elif kind == "serve":
        most = 400
    else:
        most = min(100000, 4e9 / (hits * shape[0]))
    case["windows"] = max(1, int(_log(rng, 1 if kind in ("find", "serve") else 100,
                                      max(most, 101))))
    return case


def _mean_tracks(case):
    n = case["tracks"]
    if case["law"] == "uniform":
        return (n + 1) / 2
    if case["law"] == "rate":                      # tracks per ns, windows of 10 ns
        return n * STEP_PS * OVERLAP / 1000
    return float(n)


def _hits_per_window(case):
    return _mean_tracks(case) * HITS_PER_TRACK[case["turns"]] * (1 + case["noise"])


def work(case):
    """Bytes read and written once, and the arithmetic of the votes (two
    multiply-adds a vote), for the expected number of hits."""
    W = case["windows"]
    hits = W * _hits_per_window(case)
    cells = case["n_theta"] * case["n_rho"]
    if case["kind"] == "coarse_fine":
        return {"bytes": 12 * hits + 40 * W, "flops": 4 * hits * 28}
    flops = 4 * hits * case["n_theta"]
    if case["kind"] == "accumulate":
        return {"bytes": 8 * hits + 12 * W + 4 * W * cells, "flops": flops}
    if case["kind"] == "iterative":
        tracks = _mean_tracks(case)
        return {"bytes": 12 * hits + 16 * W * (1 + tracks), "flops": flops * max(1, tracks / 2)}
    # hits in, hit_track and track_hits out, peaks of about 1.3 a track
    size = 16 * hits + 20 * W + 16 * W * min(MAX_PEAKS, 1.3 * _mean_tracks(case))
    if case["kind"] == "export":
        size += 4 * W * cells
    if case["kind"] == "stream":                   # times and hits in, windows and index out
        size += 16 * hits / OVERLAP + 16 * hits + 8 * hits + 16 * W * _mean_tracks(case)
    return {"bytes": size, "flops": flops}


def exact(case, seed):
    """No output is a rounded number: all are integers, held to equality."""
    return None


# ---------------------------------------------------------------- inputs

def _hits(case, seed, dev):
    """Hits of pileup windows as the synthetic detector gives them: each
    window's tracks are generated helices, turned by a whole number of vanes
    (the detector's symmetry), plus uniform noise, in random order.  Returns
    (vane, strip, window or time of each hit)."""
    turns, stream = case["turns"], case["kind"] == "stream"
    pool = synth.generate(POOL_TRACKS, 1, (50.0, 300.0) if turns == 4 else (100.0, 300.0), 0.0,
                          seed=seed, max_turns=turns)
    g = torch.Generator(device=dev).manual_seed(seed)
    host = np.random.default_rng(seed)

    def ints(lo, hi, n):
        return torch.randint(lo, hi, (n,), generator=g, device=dev)

    W, n = case["windows"], case["tracks"]
    if stream:
        span = max(W - 2, 1) * STEP_PS
        owner = ints(0, span, round(n * span / 1000))                          # decay times
    else:
        count = {"fixed": lambda: np.full(W, n), "uniform": lambda: host.integers(1, n + 1, W),
                 "poisson": lambda: np.clip(host.poisson(n, W), 1, 40)}[case["law"]]()
        owner = torch.repeat_interleave(torch.arange(W, device=dev),
                                        torch.from_numpy(count.astype(np.int64)).to(dev))
    start = torch.from_numpy(pool.offsets).to(dev)
    track, turn = ints(0, POOL_TRACKS, len(owner)), ints(0, synth.N_VANES, len(owner))
    length = start[track + 1] - start[track]
    of = torch.repeat_interleave(torch.arange(len(owner), device=dev), length)
    first = torch.cumsum(length, 0) - length
    src = start[track][of] + torch.arange(len(of), device=dev) - first[of]
    vane = (torch.from_numpy(pool.vane).to(dev)[src] + turn[of]) % synth.N_VANES
    strip = torch.from_numpy(pool.strip).to(dev)[src]
    key = owner[of]
    n_noise = round(case["noise"] * len(of))
    if stream:
        key = key + ints(0, 2000, len(of))
        # as many hits whatever the seed: the noise makes up the difference
        total = round(len(owner) * HITS_PER_TRACK[1] * (1 + case["noise"]))
        n_noise = max(0, total - len(of))
        noise = ints(0, span + 2000, n_noise)
    else:
        noise = ints(0, W, n_noise)
    vane = torch.cat([vane, ints(0, synth.N_VANES, n_noise)])
    strip = torch.cat([strip, ints(0, synth.N_Z_STRIPS, n_noise)])
    key = torch.cat([key, noise])
    order = torch.randperm(len(key), generator=g, device=dev)
    if stream:
        order = order[:total]
    order = order[torch.sort(key[order], stable=True)[1]]
    return vane[order].int(), strip[order].int(), key[order]


class State:
    """What a program keeps: the finder, the graph plan or server over it,
    the inputs and the output buffers."""

    finder = plan = server = None

    def close(self):
        if self.server:
            self.server.close()
        if self.plan:
            hough.hough_plan_destroy(self.plan)
        if self.finder:
            self.finder.close()
        self.server = self.plan = self.finder = None

    def __del__(self):
        self.close()


def prepare(case, seed):
    dev = "cuda"
    s = State()
    s.case, s.kind, W = case, case["kind"], case["windows"]
    vane, strip, key = _hits(case, seed, dev)
    n = len(vane)
    # per-hit outputs sized for the largest batch a program expects
    room = n * OVERLAP if s.kind == "stream" else int(2 * W * _hits_per_window(case)) + 2000
    f = s.finder = hough.Finder(case["n_theta"], case["n_rho"], max_peaks=MAX_PEAKS,
                                export_acc=s.kind == "export")
    s.hits = dict(vane=vane, strip=strip)
    if case["encoded"]:
        s.hits = dict(phi_q=torch.empty_like(vane), z_q=torch.empty_like(vane))
        hough.hough_encode(f.ctx, vane, strip, s.hits["phi_q"], s.hits["z_q"])

    def zeros(*shape):
        return torch.zeros(shape, dtype=torch.int32, device=dev)

    if s.kind == "stream":
        s.t = key
        s.out = f.alloc_outputs(W, room)
        s.ext = dict(tracks=zeros(W, MAX_PEAKS, 4), ext_track=zeros(room), ext_hits=zeros(room),
                     window_status=zeros(W))
        return s
    s.offsets = torch.zeros(W + 1, dtype=torch.int64, device=dev)
    s.offsets[1:] = torch.cumsum(torch.bincount(key, minlength=W), 0)
    if s.kind == "serve":
        s.arrays = [x.cpu().pin_memory().numpy() for x in s.hits.values()]
        s.offsets = s.offsets.cpu().pin_memory().numpy()
        s.out = {k: v.numpy() for k, v in f.alloc_outputs(W, room, device="cpu", pin=True).items()}
        s.server = hough.Server(f, n_slots=4, raw_hits=not case["encoded"])
    elif s.kind == "accumulate":
        s.out = dict(acc=zeros(W, case["n_theta"], case["n_rho"]), window_status=zeros(W))
    elif s.kind == "iterative":
        s.out = dict(tracks=zeros(W, MAX_TRACKS, 4), n_tracks=zeros(W), hit_track=zeros(room),
                     window_status=zeros(W))
    elif s.kind == "coarse_fine":
        s.out = dict(lines=zeros(W, 8), hit_track=zeros(room))
    else:
        s.out = f.alloc_outputs(W, room)
        if s.kind == "plan":
            s.plan = f.plan(s.hits, s.offsets, s.out)
    return s


def run(s):
    f, W = s.finder, s.case["windows"]
    if s.kind in ("find", "export"):
        return f.find(s.hits, s.offsets, s.out)
    if s.kind == "plan":
        hough.hough_plan_launch(s.plan)
        return s.out
    if s.kind == "accumulate":
        return f.accumulate(s.hits, s.offsets, s.out)
    if s.kind == "iterative":
        o = s.out
        hough.hough_find_iterative(f.ctx, f.hits_struct(s.hits), s.offsets, W, MAX_TRACKS,
                                   o["tracks"], o["n_tracks"], o["hit_track"],
                                   o["window_status"])
        return o
    if s.kind == "coarse_fine":
        hough.hough_find_coarse_fine(f.ctx, f.hits_struct(s.hits), s.offsets, W, s.out["lines"],
                                     s.out["hit_track"])
        return s.out
    if s.kind == "serve":
        s.server.wait(s.server.submit(*s.arrays, s.offsets, s.out))
        # entries past a window's own peaks are unspecified: take its peaks
        own = np.arange(MAX_PEAKS) < s.out["n_peaks"][:, None]
        return dict(s.out, peaks=s.out["peaks"] * own[:, :, None])
    # from one step before the first hit: every hit is in two windows
    r = f.time_slice(s.t, s.hits, -STEP_PS, STEP_PS, OVERLAP * STEP_PS, W)
    f.find(r["hits"], r["offsets"], s.out)
    f.extend(r["hits"], r["offsets"], s.out, EXT_TOL, s.ext)
    return dict(sliced=r["hits"], index=r["index"], offsets=r["offsets"], status=r["status"],
                found=s.out, extended=s.ext)
