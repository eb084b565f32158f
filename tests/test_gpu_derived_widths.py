"""Widths whose images are sums of another width's images against plans that
search each width alone.

In a plan whose widths hold {b, 2b, 4b, 8b, 16b}, only the images of width b are
transformed (two levels above 2048^2); a plan of one width transforms every image.  Both must give the
same statistics.  An image's FP32 error is of order 3e-7 sigma RMS and 6 times
that over a few million pixels, on either side, and a peak is at least 3
sigma, so peaks agree to 1e-6 relative; 2e-5 is asked for.  Where the pixel
differs, the other pixel must hold the same value within that bound.  Sizes:
transforms of a part of a warp, one warp, two warps split and several warps;
groups of 32 with 1, 2 and 3 images over; every pattern of present and absent
widths, unsorted and repeated ones; both edge rules, FP16, clipped noise.
"""

import numpy as np
import pytest

import oracle
import synth
import paper_1802_03084_gb300 as rf
from gpu_common import plans_for, small_random_segment

pytestmark = pytest.mark.gpu

RTOL = 2e-5


@pytest.fixture(scope="module", autouse=True)
def engine():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1802_03084_gb300.build import build
    build()
    rf.lib()
    torch.cuda.init()
    yield


@pytest.mark.parametrize("npix,nint,dts,partial,flags", [
    (16, 9, [1, 2, 4], False, 0),
    (32, 39, [1, 2], True, 0),
    (64, 47, [1, 2, 4], False, 0),
    (64, 71, [1, 2, 4, 8, 16, 32], True, rf.RF_NOISE_CLIPPED),
    (128, 41, [4, 1], True, rf.RF_STORE_FP16),
    (256, 67, [2, 1, 2, 4, 6, 3, 12], False, 0),
    (512, 38, [2, 4, 8], True, rf.RF_NOISE_CLIPPED | rf.RF_STORE_FP16),
    (1024, 39, [1, 2, 4], False, 0),
    (1024, 21, [1, 3, 4, 2], True, rf.RF_NOISE_CLIPPED),
    (2048, 23, [1, 2, 4, 8], True, rf.RF_STORE_FP16),
    (2048, 18, [1, 4], True, rf.RF_NOISE_CLIPPED),
    (4096, 14, [1, 2, 4], True, 0),
    (8192, 7, [1, 2, 4], True, 0),
    (64, 66, [1, 16], False, 0),
    (128, 47, [1, 2, 4, 8, 16], True, rf.RF_NOISE_CLIPPED),
    (256, 100, [3, 6, 12, 24, 48], False, 0),
    (512, 37, [1, 8, 3], True, rf.RF_STORE_FP16),
    (1024, 49, [16, 1, 2, 8], False, 0),
    (1024, 32, [1, 16], True, rf.RF_NOISE_CLIPPED),
    (2048, 33, [1, 4, 16, 8], True, rf.RF_STORE_FP16),
    (2048, 17, [1, 8, 2], False, rf.RF_NOISE_CLIPPED),
])
def test_derived_widths_equal_widths_alone(npix, nint, dts, partial, flags):
    rng = np.random.default_rng(npix + nint)
    nant, nchan, ndm = 6, 5, 3
    seg = small_random_segment(rng, nant, nchan, nint, npix)
    umax = 600.0 * seg["freq_hz"].max() / oracle.C_LIGHT
    flags |= rf.RF_EDGE_PARTIAL if partial else 0

    def plan(widths):
        spec = synth.SegmentSpec(name="w", nchan=nchan, f_lo_hz=1e9, bw_hz=1e9, nint=nint, inttime_s=2e-3, npix=npix,
                                 dm_list=np.linspace(0, 20.0, ndm), dt_list=widths, threshold=3.0, nant=nant,
                                 cell_rad=0.47 / umax)
        return plans_for(spec, seg, flags=flags)[0]

    with plan(dts) as gp:
        cands, stats = gp.search_stats(seg["vis"])
        assert len(stats) == gp.count_images(nint)
        assert np.array_equal(np.sort(stats, order=["dm_idx", "dt_idx", "t_idx"]), stats)
        gp.set_overlap(True)     # halves of the scratch, and no graph
        gp.set_graphs(False)
        c2, s2 = gp.search_stats(seg["vis"])
        assert s2.tobytes() == stats.tobytes() and np.array_equal(c2, cands)
        assert np.array_equal(gp.search(seg["vis"]), cands)
    for k, dt in enumerate(dts):
        mine = stats[stats["dt_idx"] == k]
        with plan([dt]) as one:
            alone = one.search_stats(seg["vis"])[1]
            assert len(mine) == len(alone)
            for f in ("dm_idx", "t_idx", "weight"):
                assert np.array_equal(mine[f], alone[f]), (dt, f)
            # a pixel on the clipping boundary may fall on either side: 25 / N^2 of the variance each
            stol = RTOL + (40.0 / npix ** 2 if flags & rf.RF_NOISE_CLIPPED else 0.0)
            assert np.allclose(mine["peak"], alone["peak"], rtol=RTOL, atol=0), dt
            assert np.allclose(mine["sigma"], alone["sigma"], rtol=stol, atol=0), dt
            for a, b in zip(mine, alone):
                if (a["x"], a["y"]) != (b["x"], b["y"]):
                    img = one.render(seg["vis"], [(int(b["dm_idx"]), 0, int(b["t_idx"]))])[0]
                    assert abs(img[a["y"], a["x"]] - b["peak"]) <= RTOL * abs(b["peak"]), (dt, a, b)
