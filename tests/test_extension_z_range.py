"""Track extension at the ends of the z range: geometries whose predictions and
bends pass 2^31, where 32-bit arithmetic would take hits 2^32 away for near
ones, and the widest geometry that the 32-bit kernel takes.  The find step's
outputs are made by hand (every hit of a line in its peak), since no table of
such a geometry resolves lines."""
import numpy as np
import pytest

import oracle
from paper_2511_02742_gb300 import synth

pytestmark = pytest.mark.gpu
G = synth.GEOMETRY
MAX_TOL = (1 << 19) - 1
N_STRIPS = 4094
# strips of 2^20 units over the whole int32 range, and of 2^16 units over
# -2^27 < z < 2^27
WIDE = dict(G, n_z_strips=N_STRIPS, z_pitch_u=1 << 20, z_min_u=-(1 << 31), z_u_per_mm=1 << 23)
NARROW = dict(G, n_z_strips=N_STRIPS, z_pitch_u=1 << 16, z_min_u=-(1 << 27) + (1 << 16),
              z_u_per_mm=1 << 19)


def _windows():
    """Lists of (vane, strip) per peak, of each window."""
    rng = np.random.default_rng(81)
    # a bend of -2^32, no seed; extrapolations 4096 strips off, forward and
    # backward; a line all round
    parts = [[[(0, 0), (1, 2048), (2, 0)]],
             [[(5, 1000), (6, 2500), (7, 4000), (8, 5500 - 4096)]],
             [[(5, 4000 - 4096 + 1500), (6, 4000), (7, 2500), (8, 1000)]],
             [[(v, 90 + 100 * v) for v in range(40)]]]
    for _ in range(40):                              # lines that leave one end and come in at the other
        peaks = []
        for _ in range(rng.integers(1, 4)):
            first, n = rng.integers(40), rng.integers(3, 41)
            s = rng.integers(4096) + rng.integers(-1600, 1600) * np.arange(n)
            peaks.append([((first + k) % 40, s[k] % 4096) for k in range(n) if s[k] % 4096 < N_STRIPS])
        parts.append(peaks)
    return parts


def _found(parts, max_peaks):
    n_hits = sum(len(p) for w in parts for p in w)
    n_w = len(parts)
    vane, strip = np.zeros(n_hits, np.int32), np.zeros(n_hits, np.int32)
    offs = np.zeros(n_w + 1, np.int64)
    peaks = np.zeros((n_w, max_peaks), oracle.PEAK_DTYPE)
    n_peaks = np.zeros(n_w, np.int32)
    hit_track, track_hits = np.zeros(n_hits, np.int32), np.zeros(n_hits, np.int32)
    at = 0
    for k, w in enumerate(parts):
        beg = at
        for p, hits in enumerate(w):
            peaks[k, p]["hit_begin"], peaks[k, p]["n_hits"] = at - beg, len(hits)
            for v, s in hits:
                vane[at], strip[at], hit_track[at], track_hits[at] = v, s, p, at - beg
                at += 1
        n_peaks[k], offs[k + 1] = len(w), at
    return vane, strip, offs, dict(peaks=peaks, n_peaks=n_peaks, hit_track=hit_track,
                                   track_hits=track_hits)


@pytest.mark.parametrize("raw", [True, False])
@pytest.mark.parametrize("geom", [WIDE, NARROW], ids=["wide", "narrow"])
def test_ends_of_the_z_range(hough, geom, raw):
    import torch
    parts = _windows()
    vane, strip, offs, found = _found(parts, 8)
    phi, z = oracle.encode(geom, vane, strip)
    re, rt, rh = oracle.extend(geom, phi, z, offs, found, MAX_TOL)
    assert re[0][0]["n_hits"] == 0                   # no seed
    assert (re[1:3, 0]["n_hits"] == 3).all() and re[3][0]["n_hits"] == 40
    if geom is WIDE:
        # what these windows are for: sums that are 0 mod 2^32, and are not 0
        z64 = z.astype(np.int64)
        assert z64[0] - 2 * z64[1] + z64[2] == -(1 << 32)
        assert (3 * z64[5] - 3 * z64[4] + z64[3]) - z64[6] == 1 << 32
        assert (3 * z64[8] - 3 * z64[9] + z64[10]) - z64[7] == 1 << 32
    else:
        assert np.abs(z).max() > (1 << 27) - (1 << 18) and geom["z_min_u"] > -(1 << 27)
        assert geom["z_min_u"] + N_STRIPS * geom["z_pitch_u"] < 1 << 27
    f = hough.Finder(64, 64, geometry=geom, max_peaks=8)
    dev = {k: torch.from_numpy(v).cuda() for k, v in found.items() if k != "peaks"}
    dev["peaks"] = torch.from_numpy(found["peaks"].view(np.int32).reshape(len(parts), 8, 4)).cuda()
    dev["n_found"] = dev["n_peaks"].clone()
    dev["window_status"] = torch.zeros(len(parts), dtype=torch.int32, device="cuda")
    hits = (dict(vane=torch.from_numpy(vane).cuda(), strip=torch.from_numpy(strip).cuda()) if raw else
            dict(phi_q=torch.from_numpy(phi).cuda(), z_q=torch.from_numpy(z).cuda()))
    out = f.extend(hits, torch.from_numpy(offs).cuda(), dev, MAX_TOL)
    torch.cuda.synchronize()
    ext = out["tracks"].cpu().numpy().view(hough.EXT_DTYPE).reshape(len(parts), 8)
    for k, w in enumerate(parts):
        np.testing.assert_array_equal(ext[k][:len(w)], re[k][:len(w)], err_msg=str(k))
    np.testing.assert_array_equal(out["ext_track"].cpu().numpy()[:len(vane)], rt)
    np.testing.assert_array_equal(out["ext_hits"].cpu().numpy()[:len(vane)], rh)
    assert (out["window_status"].cpu().numpy() == 0).all()
    f.close()
