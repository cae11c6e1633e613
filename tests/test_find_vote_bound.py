"""The find's vote bound in windows of 256 hits and more: it is taken from the
live histogram while other warps append, by one look for the whole warp, and
drops only peaks that cannot be kept.  Bit for bit against the oracle, again
and again, with few to many kept peaks and in every CTA size."""
import numpy as np
import pytest

from parity_helpers import assert_batch_equal, gpu_run, oracle_run
from test_find_edges import _random, _windows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("max_peaks", [0, 1, 2, 31, 64, 256])
def test_bound_from_the_live_histogram(hough, max_peaks):
    rng = np.random.default_rng(31)
    w = _windows([_random(rng, n) for n in (256, 300, 500, 1000, 1023) for _ in range(4)])
    ref = oracle_run(w, 512, 512, vote_threshold=2, max_peaks=max_peaks)
    assert (ref["n_found"] > 2000).all()
    f = hough.Finder(512, 512, vote_threshold=2, max_peaks=max_peaks)
    for shape in ((0, 0, 0, 0), (128, 32, 512, 1), (512, 32, 1024, 2), (1024, 32, 1024, 1)):
        hough.hough_set_launch(f.ctx, *shape)
        for _ in range(4):
            assert_batch_equal(gpu_run(f, w), ref, w)
    f.close()
