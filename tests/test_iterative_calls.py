"""The iterative search beside other work of its context: nothing of a call is
shared with a find that was captured on its stream, and a call needs no memory
of the library's own."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2511_02742_gb300 import synth

pytestmark = pytest.mark.gpu

MAX_TRACKS = 16


class _Search:
    """Windows on the GPU, their iterative search, and the oracle's answer."""

    def __init__(self, hough, n_windows, seed):
        import torch
        self.hough = hough
        self.w = synth.generate(n_windows, ("poisson", 6, 0, 30), (100.0, 300.0), 0.02, seed=seed)
        self.f = hough.Finder(256, 256)
        self.hits = dict(vane=torch.from_numpy(self.w.vane).cuda(),
                         strip=torch.from_numpy(self.w.strip).cuda())
        self.offs = torch.from_numpy(self.w.offsets).cuda()

    def outputs(self):
        import torch
        n = self.w.n_windows
        return (torch.full((n, MAX_TRACKS, 4), -7, dtype=torch.int32, device="cuda"),
                torch.full((n,), -7, dtype=torch.int32, device="cuda"),
                torch.full((self.w.n_hits,), -7, dtype=torch.int32, device="cuda"),
                torch.full((n,), -7, dtype=torch.int32, device="cuda"))

    def call(self, out, stream):
        self.hough.hough_find_iterative(self.f.ctx, self.f.hits_struct(self.hits), self.offs,
                                        self.w.n_windows, MAX_TRACKS, *out, stream=stream)

    def check(self, *outs):
        w = self.w
        phi, z = oracle.encode(synth.GEOMETRY, w.vane, w.strip)
        rtr, rnt, rht = oracle.iterative(synth.GEOMETRY, 256, 256, phi, z, w.offsets,
                                         max_tracks=MAX_TRACKS)
        for tr, nt, ht, st in outs:
            tr = tr.cpu().numpy().view(self.hough.ITER_DTYPE).reshape(w.n_windows, MAX_TRACKS)
            np.testing.assert_array_equal(nt.cpu().numpy(), rnt)
            for k in range(w.n_windows):
                np.testing.assert_array_equal(tr[k][:rnt[k]], rtr[k][:rnt[k]], err_msg=str(k))
            np.testing.assert_array_equal(ht.cpu().numpy(), rht)
            assert (st.cpu().numpy() == 0).all()


def test_beside_a_find_captured_on_its_stream(hough):
    """A find captured on stream a is replayed on stream b while the search
    runs on a: both give the oracle's results, and so do later calls on a."""
    import torch
    s = _Search(hough, 3000, 44)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    found, again = (s.f.alloc_outputs(s.w.n_windows, s.w.n_hits) for _ in range(2))
    outs = [s.outputs() for _ in range(4)]
    torch.cuda.synchronize()
    s.f.find(s.hits, s.offs, out=again, stream=a)
    a.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=a, capture_error_mode="thread_local"):
        s.f.find(s.hits, s.offs, out=found, stream=a)
    for out in outs[:3]:
        with torch.cuda.stream(b):
            g.replay()
        s.call(out, a)
    torch.cuda.synchronize()
    s.call(outs[3], a)
    torch.cuda.synchronize()
    s.check(*outs)
    for k in ("n_peaks", "n_found", "hit_track", "track_hits", "window_status"):
        np.testing.assert_array_equal(found[k].cpu().numpy(), again[k].cpu().numpy(), err_msg=k)
    s.f.close()


def test_new_stream_while_another_is_captured(hough):
    """The first call on a stream, while another stream is captured in the mode
    that forbids allocations: the search runs, and the capture stays whole."""
    import torch
    s = _Search(hough, 400, 45)
    warm, out = s.outputs(), s.outputs()
    s.call(warm, torch.cuda.current_stream())
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")
    captured, fresh = torch.cuda.Stream(), torch.cuda.Stream()
    graph = ctypes.c_void_p()
    assert cu.cuStreamBeginCapture_v2(ctypes.c_void_p(captured.cuda_stream), 0) == 0
    try:
        s.call(out, fresh)
    finally:
        ended = cu.cuStreamEndCapture(ctypes.c_void_p(captured.cuda_stream), ctypes.byref(graph))
    assert ended == 0
    assert cu.cuGraphDestroy(graph) == 0
    torch.cuda.synchronize()
    s.check(warm, out)
    s.f.close()
