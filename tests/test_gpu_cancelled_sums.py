"""Sums of images that cancel.

A width as long as a mean-subtracted segment, and integrations whose bright
interference changes sign, leave a sum far fainter than its parts.  Such images
are made from their own samples: records and candidates of a plan of many widths
against plans of each width alone, byte for byte where the sum cancels (both then
run the same kernels on the same sums), else within the bound of sums: an image's
FP32 error is of order 3e-7 sigma RMS, a sum's at most twice that where its parts
hold up to four times its power, and 6 times that over a few million pixels, so
peaks of at least 3 sigma agree to 2e-6 relative; 2e-5 is asked for.
"""

import numpy as np
import pytest

import oracle
import synth
import paper_1802_03084_gb300 as rf
from gpu_common import plans_for, small_random_segment

pytestmark = pytest.mark.gpu

RTOL = 2e-5


def _check(seg, vis, npix, dts, flags, cancels):
    nint, nchan = vis.shape[0], vis.shape[2]
    umax = 600.0 * seg["freq_hz"].max() / oracle.C_LIGHT

    def plan(widths):
        spec = synth.SegmentSpec(name="x", nchan=nchan, f_lo_hz=1e9, bw_hz=1e9, nint=nint, inttime_s=2e-3, npix=npix,
                                 dm_list=np.array([0.0]), dt_list=widths, threshold=7.0, nant=12,
                                 cell_rad=0.47 / umax)
        return plans_for(spec, seg, flags=flags)[0]

    with plan(dts) as gp:
        cands, stats = gp.search_stats(vis)
        assert gp.search(vis).tobytes() == cands.tobytes()
        assert gp.search(vis).tobytes() == cands.tobytes()  # graph replay
        gp.set_overlap(True)
        gp.set_graphs(False)
        c2, s2 = gp.search_stats(vis)
        assert c2.tobytes() == cands.tobytes() and s2.tobytes() == stats.tobytes()
        other = seg["vis"]  # nothing is kept from one search for the next
        a = gp.search_stats(other)[1]
    with plan(dts) as gp:
        assert gp.search_stats(other)[1].tobytes() == a.tobytes()
    some = False
    for k, dt in enumerate(dts):
        with plan([dt]) as one:
            calone, alone = one.search_stats(vis)
        mine = stats[stats["dt_idx"] == k]
        assert len(mine) == len(alone)
        assert len(cands[cands["dt_idx"] == k]) == len(calone), dt
        if cancels(dt):
            some = True
            for f in ("t_idx", "x", "y", "peak", "sigma", "snr", "mean", "weight"):
                assert mine[f].tobytes() == alone[f].tobytes(), (dt, f)
        else:
            stol = RTOL + (40.0 / npix ** 2 if flags & rf.RF_NOISE_CLIPPED else 0.0)
            assert np.allclose(mine["peak"], alone["peak"], rtol=RTOL, atol=0), dt
            assert np.allclose(mine["sigma"], alone["sigma"], rtol=stol, atol=0), dt
    assert some


@pytest.mark.parametrize("npix,dts,flags", [
    (64, [1, 2, 4], 0), (64, [1, 2, 4, 8, 16], rf.RF_NOISE_CLIPPED), (256, [1, 2, 4, 8], rf.RF_EDGE_PARTIAL),
    (512, [2, 4, 8], 0), (1024, [1, 2, 4, 8], 0), (1024, [1, 4], rf.RF_NOISE_CLIPPED),
    (2048, [1, 2, 4, 8, 16], 0), (2048, [1, 2], rf.RF_EDGE_PARTIAL), (4096, [1, 2, 4], 0),
])
def test_width_as_long_as_a_mean_subtracted_segment(npix, dts, flags):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    nint = dts[-1]
    seg = small_random_segment(np.random.default_rng(npix + nint), 12, 8, nint, npix)
    _check(seg, seg["vis"], npix, dts, flags | rf.RF_MEAN_SUBTRACT, lambda dt: dt == nint)


@pytest.mark.parametrize("npix,dts,flags", [
    (64, [1, 2, 4], 0), (128, [1, 2, 4, 8, 16], rf.RF_NOISE_CLIPPED), (512, [1, 2, 4], rf.RF_EDGE_PARTIAL),
    (1024, [1, 2, 4, 8], 0), (2048, [1, 2, 4, 8, 16], 0), (2048, [1, 4], 0), (4096, [1, 2], 0),
])
def test_interference_that_changes_sign(npix, dts, flags):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    rng = np.random.default_rng(npix + len(dts))
    nint = 38
    seg = small_random_segment(rng, 12, 8, nint, npix)
    phase = np.exp(2j * np.pi * rng.uniform(size=seg["vis"].shape[1:3]))
    sign = (-1.0) ** np.arange(nint)
    bad = (1e5 * sign)[:, None, None, None] * phase[None, :, :, None]
    vis = (seg["vis"] + bad).astype(np.complex64)
    _check(seg, vis, npix, dts, flags, lambda dt: dt > 1)
