"""An image does not depend on the images beside it.

In a plan with widths 8 or 16 times another, the row pass takes the same row of
two consecutive images in one transform.  Integrations that are saturated,
empty, or hold a NaN or an infinity change the images that contain them and no
other one: the records of a plan of many widths against those of a plan of the
one width, whose transforms hold rows of one image only.

An image's FP32 error is of order 3e-7 sigma RMS, on either side, and 6 times
that over a few million pixels; beside an image at most 1.5 times as bright, 1.3
times that again.  A peak is at least 3 sigma, so peaks agree to 1e-6 relative;
2e-5 is asked for, and the lower pixel of two equal ones may be the other one.
"""

import numpy as np
import pytest

import oracle
import synth
import paper_1802_03084_gb300 as rf
from gpu_common import plans_for, small_random_segment

pytestmark = pytest.mark.gpu

RTOL = 2e-5


@pytest.mark.parametrize("npix,dts,flags", [
    (64, [1, 2, 4, 8], 0),
    (128, [1, 8], rf.RF_NOISE_CLIPPED),
    (256, [1, 2, 4, 8, 16], rf.RF_EDGE_PARTIAL),
    (512, [1, 16], 0),
    (1024, [1, 2, 4, 8], 0),
    (1024, [1, 4, 8, 16], rf.RF_NOISE_CLIPPED | rf.RF_EDGE_PARTIAL),
    (2048, [1, 2, 4, 8, 16], 0),
    (2048, [1, 8, 2], rf.RF_EDGE_PARTIAL),
    (1024, [1, 2, 4], 0),       # two rows of one image a transform
])
def test_neighbours_of_bad_integrations(npix, dts, flags):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    rng = np.random.default_rng(npix + len(dts))
    nint, nchan = 43, 5
    seg = small_random_segment(rng, 6, nchan, nint, npix)
    umax = 600.0 * seg["freq_hz"].max() / oracle.C_LIGHT
    vis = seg["vis"]
    vis[2] *= 1.4               # still beside its neighbour in one transform
    vis[7] *= 1e6
    vis[12] *= 1e9
    vis[16:18] = 0
    vis[20] = 0
    vis[25, 3, 2, 0] = np.nan
    vis[30, 1, 4, 1] = np.inf
    vis[34] *= 1e-6

    def plan(widths):
        spec = synth.SegmentSpec(name="c", nchan=nchan, f_lo_hz=1e9, bw_hz=1e9, nint=nint, inttime_s=2e-3, npix=npix,
                                 dm_list=np.array([0.0, 20.0]), dt_list=widths, threshold=3.3, nant=6,
                                 cell_rad=0.47 / umax)
        return plans_for(spec, seg, flags=flags)[0]

    with plan(dts) as gp:
        cands, stats = gp.search_stats(vis)
        assert gp.search(vis).tobytes() == cands.tobytes()
    for k, dt in enumerate(dts):
        mine, found = stats[stats["dt_idx"] == k], cands[cands["dt_idx"] == k]
        with plan([dt]) as one:
            calone, alone = one.search_stats(vis)
            delays = one.delays()
        # images that contain the infinity: no pixel of theirs is defined
        clean = np.array([not np.any((a["t_idx"] * dt + delays[a["dm_idx"]] <= 30) &
                                     (a["t_idx"] * dt + delays[a["dm_idx"]] + dt > 30)) for a in alone])
        assert 0 < clean.sum() < len(alone)
        stol = RTOL + (40.0 / npix ** 2 if flags & rf.RF_NOISE_CLIPPED else 0.0)
        a, b = mine[clean], alone[clean]
        assert np.allclose(a["peak"], b["peak"], rtol=RTOL, atol=0), dt
        assert np.allclose(a["sigma"], b["sigma"], rtol=stol, atol=0), dt
        same = (a["x"] == b["x"]) & (a["y"] == b["y"])
        assert same.mean() > 0.9, dt
        # the same candidates, but for those at the threshold
        key = lambda c: {(int(x["dm_idx"]), int(x["t_idx"])) for x in c if abs(x["snr"] - 3.3) > 1e-3}
        near = {(int(x["dm_idx"]), int(x["t_idx"])) for x in alone if abs(x["snr"] - 3.3) <= 1e-3}
        assert key(found) - near == key(calone) - near, dt
    assert len(cands) > 0
