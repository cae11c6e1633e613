"""A call that could not allocate says so, and the calls after it are not
charged with its error."""
import ctypes

import numpy as np
import pytest

from paper_2511_02742_gb300 import synth

pytestmark = pytest.mark.gpu


def test_find_after_a_refused_allocation(hough):
    """The first find on a stream allocates its scheduling counter, which CUDA
    refuses while another stream of the thread is captured in the global mode:
    HOUGH_ERR_ALLOC, and finds on streams that have theirs run as before."""
    import torch
    w = synth.generate(400, ("poisson", 6, 0, 30), (100.0, 300.0), 0.02, seed=46)
    f = hough.Finder(256, 256)
    hits = dict(vane=torch.from_numpy(w.vane).cuda(), strip=torch.from_numpy(w.strip).cuda())
    offs = torch.from_numpy(w.offsets).cuda()
    ref, out = f.alloc_outputs(w.n_windows, w.n_hits), f.alloc_outputs(w.n_windows, w.n_hits)
    known, fresh, captured = (torch.cuda.Stream() for _ in range(3))
    torch.cuda.synchronize()
    f.find(hits, offs, out=ref, stream=known)
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")
    graph = ctypes.c_void_p()
    assert cu.cuStreamBeginCapture_v2(ctypes.c_void_p(captured.cuda_stream), 0) == 0
    try:
        with pytest.raises(hough.HoughError) as e:
            f.find(hits, offs, out=out, stream=fresh)
    finally:
        cu.cuStreamEndCapture(ctypes.c_void_p(captured.cuda_stream), ctypes.byref(graph))
    assert e.value.code == -2                     # HOUGH_ERR_ALLOC
    if graph.value:
        cu.cuGraphDestroy(graph)
    f.find(hits, offs, out=out, stream=known)
    torch.cuda.synchronize()
    for k in ("n_peaks", "n_found", "hit_track", "track_hits", "window_status"):
        np.testing.assert_array_equal(out[k].cpu().numpy(), ref[k].cpu().numpy(), err_msg=k)
    f.close()
