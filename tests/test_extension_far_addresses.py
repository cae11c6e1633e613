"""Strip addresses so far outside the detector that their phi wraps, mod 2^32,
into it: the find takes them as their encoded phi, and so does the extension,
with vanes that are never an index past the detector's."""
import numpy as np
import pytest

import oracle
from paper_2511_02742_gb300 import synth

pytestmark = pytest.mark.gpu
G = synth.GEOMETRY
STEP = 360 * G["phi_u_per_deg"] // G["n_vanes"]
PHI_END = 360 * G["phi_u_per_deg"]


def _far(rng, n):
    """n vane addresses outside [0, n_vanes) whose phi wraps into the box."""
    turns = rng.integers(-800, 800, n)
    v = (turns * (1 << 32) + rng.integers(0, PHI_END, n) - 1) // STEP + 1
    v = v[(v < 0) | (v >= G["n_vanes"])]
    phi = (v * STEP).astype(np.int64) & 0xffffffff
    return v[phi < PHI_END].astype(np.int32)


def test_wrapped_addresses(hough):
    import torch
    rng = np.random.default_rng(82)
    w = synth.generate(60, ("poisson", 6, 1, 20), (100.0, 300.0), 0.02, seed=83)
    vane = w.vane.copy()
    # some vanes as addresses of the same phi (2^29 vane steps are whole turns of
    # 2^32), some of any phi of the box
    same = rng.random(w.n_hits) < 0.1
    vane[same] += rng.choice([-(1 << 30), -(1 << 29), 1 << 29, 1 << 30], same.sum()).astype(np.int32)
    assert (STEP << 29) % (1 << 32) == 0
    far = _far(rng, 4000)
    assert len(far) > 1000 and ((far.astype(np.int16) >= G["n_vanes"]) & (far < 0)).any()
    other = np.flatnonzero(~same)[rng.permutation((~same).sum())[:w.n_hits // 10]]
    vane[other] = far[:len(other)]
    phi, z = oracle.encode(G, vane, w.strip)
    ref = oracle.find_batch(G, 256, 256, phi, z, w.offsets, max_peaks=64)
    re, rt, rh = oracle.extend(G, phi, z, w.offsets, ref, 16 * 38)
    assert (rt[same] >= 0).any()
    f = hough.Finder(256, 256, max_peaks=64)
    hits = dict(vane=torch.from_numpy(vane).cuda(), strip=torch.from_numpy(w.strip).cuda())
    o = torch.from_numpy(w.offsets).cuda()
    found = f.find(hits, o)
    out = f.extend(hits, o, found, 16 * 38)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(found["n_peaks"].cpu().numpy(), ref["n_peaks"])
    np.testing.assert_array_equal(found["hit_track"].cpu().numpy()[:w.n_hits], ref["hit_track"])
    ext = out["tracks"].cpu().numpy().view(hough.EXT_DTYPE).reshape(w.n_windows, 64)
    for k in range(w.n_windows):
        np.testing.assert_array_equal(ext[k][:ref["n_peaks"][k]], re[k][:ref["n_peaks"][k]])
    np.testing.assert_array_equal(out["ext_track"].cpu().numpy()[:w.n_hits], rt)
    np.testing.assert_array_equal(out["ext_hits"].cpu().numpy()[:w.n_hits], rh)
    f.close()
