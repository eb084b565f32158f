"""Periodicity searches in waves that hold one group of images.

The two images of a frequency are in one wave; where a wave holds fewer images
than a block of frequencies makes, blocks are smaller.  Every record has to be
the same, byte for byte, as in waves that hold everything.  Small waves come from
the tuning knob, from a short list of images (one DM, long widths) and from both;
counts of frequencies below, at and above a block's.
"""

import numpy as np
import pytest

import oracle
import synth
from gpu_common import plans_for, small_random_segment

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npix,dts,kmin,kmax", [
    (64, [1], 1, 64), (256, [1, 2, 4], 3, 34), (512, [1], 1, 32), (512, [1], 2, 64), (1024, [1], 1, 32),
    (1024, [1], 1, 64), (1024, [1, 2, 4, 8], 5, 40), (2048, [1], 1, 33), (512, [8], 1, 47), (1024, [16], 1, 32),
])
def test_small_waves_give_the_same_records(npix, dts, kmin, kmax):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    L, nint = 128, 134
    seg = small_random_segment(np.random.default_rng(npix + kmax), 6, 5, nint, npix)
    umax = 600.0 * seg["freq_hz"].max() / oracle.C_LIGHT

    def plan(widths, dms):
        spec = synth.SegmentSpec(name="p", nchan=5, f_lo_hz=1e9, bw_hz=1e9, nint=nint, inttime_s=2e-3, npix=npix,
                                 dm_list=dms, dt_list=widths, threshold=3.0, nant=6, cell_rad=0.47 / umax)
        return plans_for(spec, seg)[0]

    dms = np.array([0.0, 1.0, 2.0])
    with plan([1], dms) as gp:
        assert gp.wave_images() >= 2 * 64
        want = gp.periodicity_search(seg["vis"], L, kmin, kmax, 4.0, with_stats=True)
        assert len(want[1]) == 3 * (kmax - kmin + 1)
    with plan(dts, dms) as gp:
        for n in (32, 33, 50, 64):
            gp.set_wave_images(n)
            got = gp.periodicity_search(seg["vis"], L, kmin, kmax, 4.0, with_stats=True)
            assert got[0].tobytes() == want[0].tobytes() and got[1].tobytes() == want[1].tobytes(), n
    with plan(dts, dms[:1]) as gp:  # as few slots as the images of the search need
        got = gp.periodicity_search(seg["vis"], L, kmin, kmax, 4.0, with_stats=True)
        assert got[1].tobytes() == want[1][want[1]["dm_idx"] == 0].tobytes()
