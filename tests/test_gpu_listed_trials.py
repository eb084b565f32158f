"""Images of listed trials gridded from the samples themselves against those
gridded from resampled series.

A few trials are summed from S, many from series resampled for all times; the
sums are formed in the same order, so the images are equal byte for byte.
Widths that do not divide the segment, sweeps past its end, FP16 storage.
"""

import numpy as np
import pytest

import oracle
import synth
import paper_1802_03084_gb300 as rf
from gpu_common import plans_for, small_random_segment

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npix,nint,dts,flags", [
    (64, 37, [1, 2, 3, 8], rf.RF_EDGE_PARTIAL),
    (256, 50, [1, 4, 5], rf.RF_STORE_FP16),
    (1024, 33, [2, 7, 32], rf.RF_EDGE_PARTIAL | rf.RF_STORE_FP16),
    (2048, 21, [1, 3], rf.RF_MEAN_SUBTRACT),
])
def test_few_trials_equal_many(npix, nint, dts, flags):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    seg = small_random_segment(np.random.default_rng(npix + nint), 6, 5, nint, npix)
    umax = 600.0 * seg["freq_hz"].max() / oracle.C_LIGHT
    spec = synth.SegmentSpec(name="l", nchan=5, f_lo_hz=1e9, bw_hz=1e9, nint=nint, inttime_s=2e-3, npix=npix,
                             dm_list=np.linspace(0, 20.0, 3), dt_list=dts, threshold=3.0, nant=6,
                             cell_rad=0.47 / umax)
    with plans_for(spec, seg, flags=flags)[0] as gp:
        stats = gp.search_stats(seg["vis"])[1]
        for s in range(len(dts)):
            mine = stats[stats["dt_idx"] == s]
            if not len(mine):
                continue
            r = mine[-1]  # the last time searched: under PARTIAL its sweep leaves the segment
            trial = (int(r["dm_idx"]), s, int(r["t_idx"]))
            few = gp.render(seg["vis"], [trial])[0]
            many = gp.render(seg["vis"], [trial] * (nint // dts[s] + 1))  # more samples than a resampled series
            assert few.tobytes() == many[0].tobytes() == many[-1].tobytes(), trial
            assert abs(few[r["y"], r["x"]] - r["peak"]) <= 2e-5 * abs(r["peak"])
