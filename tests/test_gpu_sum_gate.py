"""Candidates among sums of 2 .. 16 images, searched alone and with statistics.

Without statistics a sum's maximum is taken only where the maxima of its parts
reach its gate together, and that bound is carried up level by level.  Records
have to be the same, byte for byte, as of a search with statistics.  A weak
steady source makes the widest images the most significant ones, and thresholds
lie at S/Ns of each width's own images, up to its largest: there a sum has to be
kept at its own gate while every one of its parts is below theirs.  Lengths leave
odd last images, partial units and groups; one integration is far brighter, so
its images share no transform.
"""

import numpy as np
import pytest

import oracle
import synth
import paper_1802_03084_gb300 as rf
from gpu_common import plans_for, small_random_segment

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bright", [False, True])
@pytest.mark.parametrize("npix,nint,dts,flags", [
    (64, 81, [1, 2, 4, 8], 0), (64, 64, [1, 16], 0), (128, 51, [1, 2, 4, 8, 16], 0), (256, 83, [1, 8, 3], 0),
    (256, 47, [1, 16], 0), (512, 53, [1, 2, 4, 8, 16], rf.RF_EDGE_PARTIAL), (512, 33, [1, 8, 3], 0),
    (1024, 49, [1, 2, 4, 8], 0), (1024, 39, [1, 2, 4, 8, 16], rf.RF_STORE_FP16), (1024, 35, [1, 16], 0),
    (2048, 39, [1, 2, 4, 8, 16], 0), (2048, 35, [1, 8, 3], rf.RF_EDGE_PARTIAL), (2048, 32, [1, 16], 0),
])
def test_sums_at_their_own_gate(npix, nint, dts, flags, bright):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    rng = np.random.default_rng(npix + nint)
    seg = small_random_segment(rng, 7, 6, nint, npix)
    # a source at the phase centre, some 3 sigma in one image and 12 in a sum of 16
    shape = seg["vis"].shape
    seg["vis"] = (0.8 + 4.0 * (rng.standard_normal(shape) + 1j * rng.standard_normal(shape))).astype(np.complex64)
    umax = 600.0 * seg["freq_hz"].max() / oracle.C_LIGHT
    if bright:
        seg["vis"][nint // 3] *= 30.0

    def search(threshold):
        spec = synth.SegmentSpec(name="s", nchan=6, f_lo_hz=1e9, bw_hz=1e9, nint=nint, inttime_s=2e-3, npix=npix,
                                 dm_list=np.array([0.0, 4.0, 8.0]), dt_list=dts, threshold=threshold, nant=7,
                                 cell_rad=0.47 / umax)
        with plans_for(spec, seg, flags=flags)[0] as gp:
            cands, stats = gp.search_stats(seg["vis"])
            assert gp.search(seg["vis"]).tobytes() == cands.tobytes(), threshold
            return cands, stats

    stats = search(3.0)[1]
    alone = 0
    for k in range(len(dts)):
        snr = np.sort(stats["snr"][stats["dt_idx"] == k])
        for at in {snr[len(snr) // 2], snr[-min(2, len(snr))], snr[-1]}:
            # the record's S/N is rounded to FP32: one step below is reached for certain
            cands = search(float(np.nextafter(at, np.float32(0))))[0]
            assert 0 < len(cands) <= len(stats)
            # sums found whose parts of the base width are not
            base = {(int(c["dm_idx"]), int(c["t_idx"])) for c in cands[cands["dt_idx"] == 0]}
            alone += sum(dts[int(c["dt_idx"])] in (2, 4, 8, 16) and not any(
                (int(c["dm_idx"]), int(c["t_idx"]) * dts[int(c["dt_idx"])] + j) in base
                for j in range(dts[int(c["dt_idx"])])) for c in cands)
    # (a bright image's sums are as significant as the image)
    assert alone > 0 or bright
