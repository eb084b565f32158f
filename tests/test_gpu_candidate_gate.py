"""A search that returns candidates alone against one that returns every
image's statistics.

Without statistics the row pass leaves out the peak positions of images that
cannot be candidates; the candidates have to be the same records, byte for
byte, positions included.  Thresholds lie at an image's own S/N, where a gate
that is too high would lose it, and at one that only a few images reach.  Sizes:
transforms of a part of a warp, one warp, two warps split and several warps,
with and without widths that are sums of others.
"""

import numpy as np
import pytest

import oracle
import synth
import paper_1802_03084_gb300 as rf
from gpu_common import plans_for, small_random_segment

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npix,nint,dts", [
    (16, 70, [1]), (64, 70, [1, 2, 4]), (128, 45, [1, 3]), (256, 67, [1, 2]), (512, 41, [1]), (512, 41, [1, 2, 4]),
    (1024, 37, [1]), (1024, 37, [1, 2, 4]), (2048, 21, [1]), (2048, 21, [1, 4]), (4096, 9, [1, 2]), (4096, 5, [1]),
])
def test_candidates_alone_equal_candidates_with_statistics(npix, nint, dts):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    rng = np.random.default_rng(npix + nint + len(dts))
    seg = small_random_segment(rng, 6, 5, nint, npix)
    umax = 600.0 * seg["freq_hz"].max() / oracle.C_LIGHT

    def search(threshold, flags=0):
        spec = synth.SegmentSpec(name="g", nchan=5, f_lo_hz=1e9, bw_hz=1e9, nint=nint, inttime_s=2e-3, npix=npix,
                                 dm_list=np.linspace(0, 20.0, 3), dt_list=dts, threshold=threshold, nant=6,
                                 cell_rad=0.47 / umax)
        with plans_for(spec, seg, flags=flags)[0] as gp:
            cands, stats = gp.search_stats(seg["vis"])
            assert gp.search(seg["vis"]).tobytes() == cands.tobytes()
            return cands, stats

    snr = np.sort(search(3.0)[1]["snr"])
    for threshold in (snr[len(snr) // 2], snr[-3]):
        cands = search(float(threshold))[0]
        assert 0 < len(cands) < len(snr)
    search(float(snr[len(snr) // 2]), rf.RF_NOISE_CLIPPED)
    seg["vis"][:] = 0  # empty images: no noise, no candidate
    assert len(search(1.0)[0]) == 0
