"""Listed trials of a plan with more channels than the delays of one DM fit a
block's default shared memory (12,288): rendered from the samples and from
resampled series, and in candidate products, against FP64 images.
"""

import numpy as np
import pytest

import oracle
import synth
from gpu_common import IMG_RMS_FP32, plans_for, rel_rms, small_random_segment

pytestmark = pytest.mark.gpu


def test_listed_trials_of_many_channels():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    rng = np.random.default_rng(3)
    nant, nchan, nint, npix = 3, 12500, 12, 64
    seg = small_random_segment(rng, nant, nchan, nint, npix)
    umax = 600.0 * seg["freq_hz"].max() / oracle.C_LIGHT
    spec = synth.SegmentSpec(name="m", nchan=nchan, f_lo_hz=1e9, bw_hz=1e9, nint=nint, inttime_s=2e-3, npix=npix,
                             dm_list=np.array([0.0, 2.0]), dt_list=[1, 2], threshold=2.0, nant=nant,
                             cell_rad=0.47 / umax)
    gp, op = plans_for(spec, seg)
    with gp:
        cands, stats = gp.search_stats(seg["vis"])
        assert len(cands) > 0
        keys = [(int(r["dm_idx"]), int(r["dt_idx"]), int(r["t_idx"])) for r in stats]
        wide = [k for k in keys if k[1] == 1]
        # few images of width 2 are gridded from the samples, many (repeated) from its resampled series
        for trials in (wide[:1] + keys[:2], (wide * nint)[:len(keys)]):
            got = gp.render(seg["vis"], trials)
            S = op.stokes(seg["vis"], nint)
            for img, k in zip(got, trials):
                assert rel_rms(img, op.image(S, *k, nint=nint)[0]) < IMG_RMS_FP32, k
        feats, _, images = gp.candidate_products(seg["vis"], cands[-2:])
        assert len(feats) == 2
        for img, c in zip(images, cands[-2:]):
            k = (int(c["dm_idx"]), int(c["dt_idx"]), int(c["t_idx"]))
            assert rel_rms(img, op.image(S, *k, nint=nint)[0]) < IMG_RMS_FP32, k
