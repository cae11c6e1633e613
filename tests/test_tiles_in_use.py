"""The tiles that contexts use with 32 word rows (host only, no GPU): the find's,
the find's with the accumulator exported, and hough_accumulate's.  Every bin
that a hit of the detector box can vote in a tile's rows is stored, stored bins
lie in the accumulator, and the alignments are those the stores rely on."""
import ctypes

import numpy as np
import pytest

from paper_2511_02742_gb300 import synth
from test_tile_bins import row_reach, tiles

G = synth.GEOMETRY
SMEM_PER_SM = 228 << 10
FIND, EXPORT, ACCUMULATE = 0, 1, 2


@pytest.fixture(scope="module")
def hough():
    from paper_2511_02742_gb300 import build, hough
    build.build()
    return hough


def in_use(hough, n_theta, n_rho, use, smem=SMEM_PER_SM):
    f = hough.load().hough_tiles_in_use
    f.restype = ctypes.c_int32
    g = hough.make_geometry(G)
    nb, p_max = ctypes.c_int32(), ctypes.c_int32()
    lo = np.full((3, (n_theta + 31) // 32), -1, np.int32)
    assert f(ctypes.byref(g), n_theta, n_rho, use, ctypes.c_int64(smem), ctypes.byref(nb),
             ctypes.byref(p_max), lo.ctypes.data_as(ctypes.c_void_p)) == 0
    return nb.value, p_max.value, lo


@pytest.mark.parametrize("n_theta,n_rho", [(512, 512), (1024, 1024), (180, 1000), (97, 332),
                                           (256, 256), (33, 64), (1, 4), (64, 512), (129, 200),
                                           (192, 1000), (193, 1000), (4096, 1024), (640, 96)])
@pytest.mark.parametrize("use", [FIND, EXPORT, ACCUMULATE])
def test_every_reachable_bin_is_stored(hough, n_theta, n_rho, use):
    nb, p_max, lo = in_use(hough, n_theta, n_rho, use)
    few = n_theta <= 192 and 1 <= n_theta % 128 <= 64
    assert p_max == (2 if few and use != ACCUMULATE else 4)
    assert 4 <= nb <= n_rho and nb % 4 == 0
    if use != FIND:
        assert nb % 32 == 0 or nb == n_rho
    first_at = {FIND: 4, EXPORT: 8 if n_rho % 8 == 0 else 4,
                ACCUMULATE: 32 if n_rho % 32 == 0 else 4}[use]
    rlo, rhi = row_reach(n_theta, n_rho)
    widest = 1
    for k in range(p_max.bit_length()):
        for i, a, b in tiles(n_theta, 32, k):
            low, high = int(rlo[a:b].min()), int(rhi[a:b].max())
            first, last = max(low, 0), min(high, n_rho - 1)
            l0 = int(lo[k, i])
            assert l0 % first_at == 0 and 0 <= l0 and l0 + nb <= n_rho, (k, i, l0)
            if last >= first:
                widest = max(widest, last - first + 1)
                assert l0 <= first and last < l0 + nb, (k, i, l0, first, last)
            if low < 0:
                assert l0 == 0
    if use == FIND:
        assert nb == min((widest + 3 + 3) // 4 * 4, n_rho)


def test_the_find_uses_the_documented_layout(hough):
    """hough_tile_bins is the find's layout, but for 64-row tiles."""
    for n_theta, n_rho in [(512, 512), (1024, 1024), (97, 332), (256, 256)]:
        nb, p_max, lo = in_use(hough, n_theta, n_rho, FIND)
        dnb, dlo = hough.hough_tile_bins(G, n_theta, n_rho, 32)
        assert p_max == 4 and nb == dnb
        np.testing.assert_array_equal(lo, dlo)
    nb, p_max, _ = in_use(hough, 180, 1000, FIND)
    assert p_max == 2 and nb < hough.hough_tile_bins(G, 180, 1000, 32)[0]


def test_accumulate_keeps_all_bins_where_three_ctas_fit(hough):
    assert in_use(hough, 512, 512, ACCUMULATE)[0] == 512
    assert in_use(hough, 1024, 1024, ACCUMULATE)[0] < 1024
    assert in_use(hough, 1024, 1024, ACCUMULATE, smem=1 << 20)[0] == 1024
