"""The iterative search on its list of bins, and where it hands a window to the
search by tiles: bit for bit against the oracle at window sizes around the
8-bit limit, with lines of more hits than a byte counts, at accumulators of a
partial tile, several tiles and several CTAs per SM, with more bins than the
list holds, and past the hits it stages."""
import numpy as np
import pytest

import oracle
from paper_2511_02742_gb300 import synth
from test_find_edges import _random, _windows
from test_iterative import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_theta,n_rho", [(512, 512), (256, 256), (130, 200), (33, 64), (180, 1000),
                                           (640, 256)])
def test_window_sizes(hough, n_theta, n_rho):
    rng = np.random.default_rng(41)
    sizes = [0, 1, 5, 31, 32, 33, 254, 255, 256, 257, 700, 1025]
    _check(hough, _windows([_random(rng, n) for n in sizes]), n_theta, n_rho, max_tracks=24)


def test_lines_past_a_byte(hough):
    rng = np.random.default_rng(42)
    parts = []
    for stack in (127, 128, 200, 255, 256, 300, 600):
        v, s = _random(rng, 60)
        parts += [(np.r_[v, [7] * stack], np.r_[s, [900] * stack]), ([7] * stack, [900] * stack)]
    _check(hough, _windows(parts), 256, 256, max_tracks=16)


def test_more_bins_than_the_list_holds(hough):
    """Dense windows: the floor rises, tracks are taken, and the hits left are
    voted again; and a window of equal bins everywhere."""
    rng = np.random.default_rng(43)
    parts = [_random(rng, n) for n in (400, 600, 900, 1000)]
    parts.append((np.repeat(np.arange(40), 6), np.tile([0, 400, 800, 1200, 1600, 2000], 40)))
    _check(hough, _windows(parts), 512, 512, max_tracks=40)
    _check(hough, _windows(parts[:3]), 1024, 1024, max_tracks=12)


def test_past_the_stage(hough):
    rng = np.random.default_rng(44)
    w = _windows([_random(rng, n) for n in (20, 1270, 2000, 2100, 3500, 4096)] +
                 [_random(rng, 30) for _ in range(30)])
    _check(hough, w, 256, 256, max_tracks=4)
    _check(hough, w, 512, 512, max_tracks=2)


def test_captured_call_beside_the_stream(hough):
    """A captured search replayed on one stream while the stream it was captured
    on runs the same calls: every result is the oracle's."""
    import torch
    w = synth.generate(3000, ("poisson", 6, 0, 30), (100.0, 300.0), 0.02, seed=44)
    f = hough.Finder(256, 256)
    hits = dict(vane=torch.from_numpy(w.vane).cuda(), strip=torch.from_numpy(w.strip).cuda())
    offs = torch.from_numpy(w.offsets).cuda()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()

    def outputs():
        return (torch.zeros((w.n_windows, 16, 4), dtype=torch.int32, device="cuda"),
                torch.zeros(w.n_windows, dtype=torch.int32, device="cuda"),
                torch.zeros(w.n_hits, dtype=torch.int32, device="cuda"),
                torch.zeros(w.n_windows, dtype=torch.int32, device="cuda"))

    def call(out, stream):
        hough.hough_find_iterative(f.ctx, f.hits_struct(hits), offs, w.n_windows, 16, *out,
                                   stream=stream)

    own, captured = outputs(), outputs()
    found = f.alloc_outputs(w.n_windows, w.n_hits)
    torch.cuda.synchronize()
    with torch.cuda.stream(a):
        f.find(hits, offs, out=found, stream=a)      # the stream has its counter
    a.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=a, capture_error_mode="thread_local"):
        call(captured, a)
    for _ in range(4):
        with torch.cuda.stream(b):
            g.replay()
        call(own, a)
        f.find(hits, offs, out=found, stream=a)
    torch.cuda.synchronize()
    phi, z = oracle.encode(synth.GEOMETRY, w.vane, w.strip)
    rtr, rnt, rht = oracle.iterative(synth.GEOMETRY, 256, 256, phi, z, w.offsets, max_tracks=16)
    for tr, nt, ht, st in (own, captured):
        tr = tr.cpu().numpy().view(hough.ITER_DTYPE).reshape(w.n_windows, 16)
        np.testing.assert_array_equal(nt.cpu().numpy(), rnt)
        for k in range(w.n_windows):
            np.testing.assert_array_equal(tr[k][:rnt[k]], rtr[k][:rnt[k]], err_msg=str(k))
        np.testing.assert_array_equal(ht.cpu().numpy(), rht)
        assert (st.cpu().numpy() == 0).all()
    f.close()
