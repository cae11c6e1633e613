"""Time slicing in blocks of every size that the library picks: window counts
around the blocks' edges, overlaps that raise the smallest block, more blocks
than run at once, against the oracle's definition."""
import numpy as np
import pytest

import oracle
from paper_2511_02742_gb300 import synth
from test_time_slice import _slice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 2, 3, 4, 5, 8, 9, 16])
@pytest.mark.parametrize("windows", [1, 7, 8, 9, 15, 16, 17, 63, 1000, 9727, 9728, 21000])
def test_windows_and_overlaps(hough, m, windows):
    rng = np.random.default_rng(100 * m + windows)
    step, n = 40, 2 * min(windows, 3000) + 5
    t = np.sort(rng.integers(-3 * step, (windows + m + 2) * step, n)).astype(np.int64)
    t[n // 2:n // 2 + 3] = t[n // 2]                       # equal times
    t = np.sort(t)
    s = synth.TimedHits(t, rng.integers(0, 40, n).astype(np.int32),
                        rng.integers(0, 2048, n).astype(np.int32), np.zeros(n, np.int64))
    f = hough.Finder(256, 256)
    r = _slice(f, s, 0, step, m * step, windows)
    offs, idx = oracle.time_slice(t, 0, step, m * step, windows)
    np.testing.assert_array_equal(r["offsets"].cpu().numpy(), offs)
    np.testing.assert_array_equal(r["index"].cpu().numpy()[:len(idx)], idx)
    np.testing.assert_array_equal(r["hits"]["vane"].cpu().numpy()[:len(idx)], s.vane[idx])
    np.testing.assert_array_equal(r["hits"]["strip"].cpu().numpy()[:len(idx)], s.strip[idx])
    assert int(r["status"].item()) == 0
    f.close()
