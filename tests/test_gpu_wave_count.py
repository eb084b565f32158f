"""A search whose transformed images fit the column-FFT scratch runs one wave.

Sweeps and remainders make the share of transformed images of a segment another
one than that of an endless one; a scratch some images short would cost a second
wave of a few images, most of a short call's time.  One gridding launch and one
column pass a search, for segments as long as the plan's and shorter ones.
"""

import numpy as np
import pytest

import oracle
import synth
import paper_1802_03084_gb300 as rf
from gpu_common import plans_for, small_random_segment

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npix,nint,ndm,dts,flags", [
    (64, 64, 2, [1, 2, 4, 8], 0), (64, 128, 4, [1, 2, 4], 0), (128, 61, 3, [1, 16], 0), (256, 64, 2, [1, 2, 4, 8], 0),
    (512, 63, 2, [1, 2, 4, 8, 16], rf.RF_EDGE_PARTIAL), (1024, 37, 2, [1, 2, 3, 6], 0), (64, 50, 5, [2, 3, 4, 12], 0),
])
def test_one_wave(npix, nint, ndm, dts, flags):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    seg = small_random_segment(np.random.default_rng(npix + nint), 6, 5, nint, npix)
    umax = 600.0 * seg["freq_hz"].max() / oracle.C_LIGHT
    spec = synth.SegmentSpec(name="w", nchan=5, f_lo_hz=1e9, bw_hz=1e9, nint=nint, inttime_s=2e-3, npix=npix,
                             dm_list=np.linspace(0, 6.0, ndm), dt_list=dts, threshold=3.0, nant=6,
                             cell_rad=0.47 / umax)
    with plans_for(spec, seg, flags=flags)[0] as gp:
        for n in (nint, nint - 1, nint // 2 + 1):
            gp.set_profiling(True)  # counts from here
            gp.search(seg["vis"][:n])
            prof = gp.profile()
            assert prof["grid_cells"][0] == prof["grid_colfft"][0] == prof["rowfft_stats"][0] == 1, (n, prof)
