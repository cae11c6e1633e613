"""Track extension over many windows of which few hold hits: a warp looks at 32
windows at a time, and each launch takes the windows of its size.  Windows of
every launch's size stand at the first, last and middle places of those looks."""
import numpy as np
import pytest

import oracle
from paper_2511_02742_gb300 import synth
from test_extension import G, TOL, _check, _oracle
from test_find_edges import _windows

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


@pytest.mark.parametrize("jitter", [0, 2, 7])
def test_tracks_that_go_round(hough, jitter):
    """Tracks on 3 to 40 of the 40 vanes, starting anywhere on the ring, alone
    and beside a second one within reach: both ends are grown at once while
    they cannot meet, and one after the other where they can."""
    rng = np.random.default_rng(91 + jitter)
    parts = []
    for n in [3, 4, 5, 20, 35, 36, 37, 38, 39, 40, 40, 39, 38]:
        for extra in (0, n // 2, 40):
            v = (rng.integers(40) + np.arange(n)) % 40
            u = (rng.integers(40) + np.arange(extra)) % 40
            vane = np.r_[v, u]
            strip = np.r_[1000 + rng.integers(-jitter, jitter + 1, n),
                          1012 + rng.integers(-jitter, jitter + 1, extra)]
            order = rng.permutation(len(vane))
            parts.append((vane[order], strip[order]))
    w = _windows(parts)
    for tol in (TOL, 40 * 38):
        _check(hough, w, 512, 512, tol=tol)


def test_wide_z(hough):
    """z of 2^27 units and more, whose predictions need 64 bits."""
    import torch
    geom = dict(G, z_pitch_u=1 << 17, z_min_u=-(1 << 27), z_u_per_mm=G["z_u_per_mm"] * 3449)
    w = synth.generate(60, ("poisson", 6, 0, 20), (100.0, 300.0), 0.05, seed=93)
    tol = (1 << 19) - 1
    f = hough.Finder(256, 256, geometry=geom, max_peaks=64)
    hits = dict(vane=torch.from_numpy(w.vane).cuda(), strip=torch.from_numpy(w.strip).cuda())
    o = torch.from_numpy(w.offsets).cuda()
    found = f.find(hits, o)
    out = f.extend(hits, o, found, tol)
    torch.cuda.synchronize()
    phi, z = oracle.encode(geom, w.vane, w.strip)
    assert np.abs(z).max() > 1 << 26
    ref = oracle.find_batch(geom, 256, 256, phi, z, w.offsets, max_peaks=64)
    re, rt, rh = oracle.extend(geom, phi, z, w.offsets, ref, tol)
    ext = out["tracks"].cpu().numpy().view(hough.EXT_DTYPE).reshape(w.n_windows, 64)
    np.testing.assert_array_equal(found["n_peaks"].cpu().numpy(), ref["n_peaks"])
    assert (rt >= 0).sum() > 100
    for k in range(w.n_windows):
        np.testing.assert_array_equal(ext[k][:ref["n_peaks"][k]], re[k][:ref["n_peaks"][k]])
    np.testing.assert_array_equal(out["ext_track"].cpu().numpy()[:w.n_hits], rt)
    np.testing.assert_array_equal(out["ext_hits"].cpu().numpy()[:w.n_hits], rh)
    f.close()


@pytest.mark.parametrize("n_windows", [300, 700, 5000])
def test_too_large_beside_others(hough, n_windows):
    """A window of more hits than a warp stages, flagged once and left without
    tracks, among windows of all sizes; the others are the oracle's."""
    import torch
    big = synth.generate(1, 330, (100.0, 300.0), 0.05, seed=94)
    w = synth.concat([synth.generate(2, t, (100.0, 300.0), 0.02, seed=95 + t) for t in (110, 50, 8)])
    n, nb = np.diff(w.offsets), int(big.offsets[1])
    assert nb > 4096
    vane = np.concatenate([w.vane, big.vane])
    strip = np.concatenate([w.strip, big.strip])
    offs = np.full(n_windows + 1, w.n_hits, np.int64)
    offs[:7] = w.offsets
    offs[n_windows] = w.n_hits + nb
    f = hough.Finder(256, 256, max_peaks=64)
    hits = dict(vane=torch.from_numpy(vane).cuda(), strip=torch.from_numpy(strip).cuda())
    o = torch.from_numpy(offs).cuda()
    found = f.find(hits, o)
    out = f.extend(hits, o, found, TOL)
    torch.cuda.synchronize()
    re, rt, rh, rnp = _oracle(w, 256, 256, TOL)
    st = out["window_status"].cpu().numpy()
    assert st[n_windows - 1] == hough.HOUGH_WIN_TOO_LARGE and (st[:n_windows - 1] == 0).all()
    ext = out["tracks"].cpu().numpy().view(hough.EXT_DTYPE).reshape(n_windows, 64)
    for k in range(6):
        np.testing.assert_array_equal(ext[k][:rnp[k]], re[k][:rnp[k]])
    et, eh = out["ext_track"].cpu().numpy(), out["ext_hits"].cpu().numpy()
    np.testing.assert_array_equal(et[:w.n_hits], rt)
    np.testing.assert_array_equal(eh[:w.n_hits], rh)
    assert (et[w.n_hits:w.n_hits + nb] == -1).all()
    np.testing.assert_array_equal(eh[w.n_hits:w.n_hits + nb], np.arange(nb))
    f.close()
