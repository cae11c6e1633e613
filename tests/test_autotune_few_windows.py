"""Autotuning on a batch of few windows, for which the library runs several CTAs
per window: the tuned context is no slower than one that was not tuned."""
import numpy as np
import pytest

from parity_helpers import assert_batch_equal, oracle_run, to_numpy
from paper_2511_02742_gb300 import synth

pytestmark = pytest.mark.gpu


def _replays_us(hough, finder, hits, offs, out):
    """GPU time of a find, from replays of a plan (no host work between them)."""
    import torch
    plan = finder.plan(hits, offs, out)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    times = []
    for _ in range(5):
        a.record()
        for _ in range(50):
            hough.hough_plan_launch(plan)
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b) * 20.0)
    hough.hough_plan_destroy(plan)
    return float(np.median(times))


@pytest.mark.parametrize("n_windows", [1, 20])
def test_tuned_is_no_slower_than_untuned(hough, n_windows):
    """1024 x 1024, 40 tracks a window: one CTA per window takes 96 to 113 us,
    several per window 35 to 48."""
    import torch
    w = synth.generate(n_windows, 40, (50.0, 300.0), 0.05, seed=17, max_turns=4)
    hits = dict(vane=torch.from_numpy(w.vane).cuda(), strip=torch.from_numpy(w.strip).cuda())
    offs = torch.from_numpy(w.offsets).cuda()
    untuned, tuned = hough.Finder(1024, 1024), hough.Finder(1024, 1024)
    out = tuned.alloc_outputs(w.n_windows, w.n_hits)
    best = tuned.autotune(hits, offs, out, iters=20)
    torch.cuda.synchronize()
    assert_batch_equal(to_numpy(out, w.n_hits), oracle_run(w, 1024, 1024), w)
    assert best == hough.hough_get_launch(tuned.ctx)
    t0, t1 = _replays_us(hough, untuned, hits, offs, out), _replays_us(hough, tuned, hits, offs, out)
    assert t1 < 1.5 * t0, (t0, t1)
    untuned.close()
    tuned.close()
