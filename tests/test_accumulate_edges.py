"""hough_accumulate at the edges of its byte counters (lines of more hits than
a byte counts, among windows of 256 hits and more), of its tiles, parts and
stage, bit for bit against the oracle."""
import numpy as np
import pytest

from test_accumulate import _check
from test_find_edges import _random, _windows
from parity_helpers import G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_theta,n_rho", [(512, 512), (1024, 1024), (180, 1000), (130, 640),
                                           (33, 36), (1, 4), (129, 992)])
def test_window_sizes_and_overflows(hough, n_theta, n_rho):
    rng = np.random.default_rng(61)
    parts = [_random(rng, n) for n in (0, 1, 33, 254, 255, 256, 700, 1023, 1024, 1025, 3000)]
    for stack in (254, 255, 256, 257, 512, 600):
        v, s = _random(rng, 90)
        parts += [(np.r_[v, [7] * stack], np.r_[s, [900] * stack]), ([7] * stack, [900] * stack)]
    _check(hough, _windows(parts), n_theta, n_rho)


def test_out_of_range_and_large(hough):
    """Votes past a narrow rho range (one part per window), and windows that
    take 16- and 32-bit counters."""
    rng = np.random.default_rng(62)
    w = _windows([_random(rng, n) for n in (20, 300, 2100, 9000)])
    _check(hough, w, 260, 256, geom=dict(G, rho_min=-120.0, rho_max=120.0))
    _check(hough, _windows([_random(rng, n) for n in (9000, 65534, 65535)]), 64, 64)
