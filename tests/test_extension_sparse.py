"""Track extension over many windows of which few hold hits: a warp looks at 32
windows at a time, and each launch takes the windows of its size.  Windows of
every launch's size stand at the first, last and middle places of those looks."""
import numpy as np
import pytest

from paper_2511_02742_gb300 import synth
from test_extension import G, TOL, _oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_windows", [1, 33, 25000, 150001])
def test_few_windows_among_empty_ones(hough, n_windows):
    import torch
    w = synth.concat([synth.generate(2, t, (100.0, 300.0), 0.02, seed=71 + t) for t in (110, 50, 8)])
    w = w.subset([0, 2, 4, 5, 3, 1]) if n_windows > 1 else w.subset([2])
    n = np.diff(w.offsets)
    assert n_windows == 1 or (n[0] > 1536 and 512 < n[1] <= 1536 and n[2] <= 512), n
    at = np.unique(np.linspace(0, n_windows - 1, w.n_windows).astype(np.int64))
    assert len(at) == w.n_windows
    offs = np.zeros(n_windows + 1, np.int64)
    offs[at + 1] = n
    offs = np.cumsum(offs)
    f = hough.Finder(256, 256, max_peaks=64)
    hits = dict(vane=torch.from_numpy(w.vane).cuda(), strip=torch.from_numpy(w.strip).cuda())
    o = torch.from_numpy(offs).cuda()
    found = f.find(hits, o)
    out = f.extend(hits, o, found, TOL)
    torch.cuda.synchronize()
    re, rt, rh, rnp = _oracle(w, 256, 256, TOL)
    n_peaks = found["n_peaks"].cpu().numpy()
    ext = out["tracks"].cpu().numpy().view(hough.EXT_DTYPE).reshape(n_windows, 64)
    np.testing.assert_array_equal(n_peaks[at], rnp)
    assert n_peaks.sum() == rnp.sum()
    for k, i in enumerate(at):
        np.testing.assert_array_equal(ext[i][:rnp[k]], re[k][:rnp[k]])
    np.testing.assert_array_equal(out["ext_track"].cpu().numpy()[:w.n_hits], rt)
    np.testing.assert_array_equal(out["ext_hits"].cpu().numpy()[:w.n_hits], rh)
    assert (out["window_status"].cpu().numpy()[:n_windows] == 0).all()
    f.close()
