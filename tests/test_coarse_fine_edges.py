"""The two-stage search at the edges of its counter widths (8 bits up to 255
hits, 16 up to 65535, then 32 with the rows in two passes) and with votes out
of the coarse range, bit for bit against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2511_02742_gb300 import synth
from test_coarse_fine import _gpu
from test_find_edges import _random, _windows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rho", [500.0, 120.0])
@pytest.mark.parametrize("raw", [True, False])
def test_window_sizes(hough, rho, raw):
    rng = np.random.default_rng(51)
    parts = [_random(rng, n) for n in (0, 1, 31, 32, 33, 200, 254, 255, 256, 257, 1000, 65535, 65536, 70000)]
    parts += [([5] * n, [1000] * n) for n in (255, 256, 300, 66000)]
    parts.append(([-1, 40, 3, 3], [5, 5, -1, 2048]))          # outside the detector box
    w = _windows(parts)
    geom = dict(synth.GEOMETRY, rho_min=-rho, rho_max=rho)
    f = hough.Finder(512, 512, geometry=geom)
    g, ght = _gpu(hough, w, raw=raw, f=f)
    f.close()
    phi, z = oracle.encode(geom, w.vane, w.strip)
    r, rht = oracle.coarse_fine(geom, phi, z, w.offsets)
    for name in oracle.CF_DTYPE.names:
        np.testing.assert_array_equal(g[name], r[name], err_msg=name)
    np.testing.assert_array_equal(ght, rht)
