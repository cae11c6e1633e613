"""The find at the edges of its counter widths, tiles and peak store, bit for
bit against the oracle: window sizes around the 8-bit limit and the packed
compares' free bit, lines of more hits than a byte counts (the window is
redone in 16 bits), accumulators of one row, of a partial tile and of one row
past a tile, every CTA size, tiles of several row groups, several CTAs per
window, stores that overflow with ties, and thresholds past a counter's range."""
import numpy as np
import pytest

from parity_helpers import assert_batch_equal, gpu_run, oracle_run
from paper_2511_02742_gb300 import synth

pytestmark = pytest.mark.gpu

SHAPES = [None, (128, 32, 256, 1), (256, 32, 512, 2), (512, 32, 512, 1), (1024, 32, 1024, 1),
          (256, 64, 512, 1), (512, 128, 512, 1)]


def _windows(parts):
    off = np.cumsum([0] + [len(v) for v, _ in parts]).astype(np.int64)
    vane = np.concatenate([np.asarray(v, np.int32) for v, _ in parts] + [np.zeros(0, np.int32)])
    strip = np.concatenate([np.asarray(s, np.int32) for _, s in parts] + [np.zeros(0, np.int32)])
    n = len(vane)
    return synth.Windows(vane.astype(np.int32), strip.astype(np.int32), off, np.zeros(n, np.int32),
                         np.zeros(n), np.zeros((0, 4)), np.zeros(len(parts) + 1, np.int64))


def _random(rng, n, spread=2048):
    """n hits, half of them along a few lines so that bins fill up."""
    v = rng.integers(0, 40, n)
    line = (rng.integers(0, 4, n) * 400 + v * 9) % spread
    return v, np.where(rng.random(n) < 0.5, line, rng.integers(0, spread, n))


def _check(hough, w, n_theta, n_rho, shapes=(None,), export=False, **th):
    ref = oracle_run(w, n_theta, n_rho, export=export, **th)
    f = hough.Finder(n_theta, n_rho, export_acc=export, **th)
    ran = 0
    for lch in shapes:
        try:
            hough.hough_set_launch(f.ctx, *(lch or (0, 0, 0, 0)))
        except hough.HoughError as e:
            assert e.code == hough.HOUGH_ERR_UNSUPPORTED_SHAPE
            continue
        assert_batch_equal(gpu_run(f, w), ref, w, check_acc=export)
        ran += 1
    f.close()
    assert ran


@pytest.mark.parametrize("n_theta,n_rho", [(512, 512), (180, 1000)])
def test_window_sizes(hough, n_theta, n_rho):
    rng = np.random.default_rng(21)
    sizes = [0, 1, 2, 3, 31, 32, 33, 63, 64, 65, 127, 128, 129, 132, 133, 254, 255, 256, 257, 511,
             512, 513, 1023, 1025, 2049]
    _check(hough, _windows([_random(rng, n) for n in sizes]), n_theta, n_rho, SHAPES)


@pytest.mark.parametrize("shape", SHAPES)
def test_lines_past_a_byte(hough, shape):
    """Stacks of 127 to 700 equal hits among others: counts with a byte's top
    bit, bins of 255 and 256, and overflows (one or several per word)."""
    rng = np.random.default_rng(22)
    parts = []
    for stack in (127, 128, 129, 200, 254, 255, 256, 257, 300, 511, 512, 700):
        v, s = _random(rng, 100)
        parts.append((np.r_[v, [7] * stack, [8] * 20], np.r_[s, [900] * stack, [900] * 20]))
        parts.append(([7] * stack, [900] * stack))
    _check(hough, _windows(parts), 256, 256, (shape,), export=True)


@pytest.mark.parametrize("n_theta,n_rho", [(1, 4), (2, 8), (31, 64), (33, 64), (127, 332),
                                           (128, 332), (129, 332), (257, 200)])
def test_small_and_partial_tiles(hough, n_theta, n_rho):
    rng = np.random.default_rng(23)
    w = _windows([_random(rng, n) for n in (40, 200, 300, 900)])
    _check(hough, w, n_theta, n_rho, SHAPES, export=True, vote_threshold=3)


@pytest.mark.parametrize("threshold", [1, 2, 128, 129, 256, 40000, 70000])
@pytest.mark.parametrize("max_peaks", [0, 1, 64, 256])
def test_thresholds_and_ties(hough, threshold, max_peaks):
    """T = 1 and 2: thousands of peaks with equal votes overflow the peak
    store; T past a byte's or a packed field's range finds only what reaches it."""
    rng = np.random.default_rng(24)
    v, s = _random(rng, 500)
    parts = [_random(rng, 150), _random(rng, 800), (np.r_[v, [3] * 300], np.r_[s, [50] * 300])]
    _check(hough, _windows(parts), 256, 512, (None, (128, 32, 512, 1), (1024, 32, 1024, 1)),
           vote_threshold=threshold, max_peaks=max_peaks)


def test_large_windows(hough):
    """Past the packed peak keys and the 8-bit attempt's hits per bin: 16-bit
    counters with 64-bit keys, and 32-bit counters."""
    rng = np.random.default_rng(25)
    w = _windows([_random(rng, n) for n in (4000, 9000, 32800, 65534, 65535, 65600)])
    _check(hough, w, 128, 128, (None, (256, 32, 512, 2)), max_peaks=16)


@pytest.mark.parametrize("n_theta,n_rho,windows", [(512, 512, 1), (512, 512, 70), (1024, 1024, 3),
                                                   (1024, 1024, 30), (257, 200, 5), (700, 300, 40)])
def test_one_window_over_several_ctas(hough, n_theta, n_rho, windows):
    """Batches of few windows run with several CTAs per window: uneven shares
    of tiles, empty windows, windows past the stage, byte overflows, and both
    wider counters; with the accumulator exported on the small ones."""
    rng = np.random.default_rng(n_theta + windows)
    sizes = [300, 0, 2500, 1, 9000, 65600, 40, 256][:windows]
    parts = [_random(rng, n) for n in sizes]
    v, s = _random(rng, 60)
    parts += [(np.r_[v, [7] * 300], np.r_[s, [900] * 300])] * (windows > 8)
    parts += [_random(rng, 20 + 7 * k) for k in range(windows - len(parts))]
    _check(hough, _windows(parts[:windows]), n_theta, n_rho, export=windows <= 5)
