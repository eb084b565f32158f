"""Device memory of plans whose widths are sums of others, as estimated before
creation (the serving runtime admits by it): no more than the images of a wave
need, and the clipped noise's partials only under RF_NOISE_CLIPPED, in the place
of the cell sums.
"""

import numpy as np
import pytest

import paper_1802_03084_gb300 as rf
from paper_1802_03084_gb300.build import build


@pytest.fixture(scope="module", autouse=True)
def library():
    build()


def _plan(npix, dts, flags=0, nint=40):
    ant = np.zeros((4, 3))
    ant[:, 0] = [0.0, 70.0, 210.0, 300.0]
    ant[:, 1] = [0.0, 120.0, -60.0, 33.0]
    f = np.array([1.2e9, 1.5e9])
    return rf.Plan(ant, f, 5e-3, npix, 0.4 / (300.0 * 1.5e9 / 299792458.0), np.array([0.0, 5.0]), dts, 7.0,
                   flags=flags | rf.RF_HOST_ONLY, max_nint=nint)


def _estimate(plan, wave=0):
    return rf.rf_plan_estimate_bytes(plan.desc, wave)


@pytest.mark.parametrize("npix", [64, 1024, 2048, 8192])
@pytest.mark.parametrize("dts", [[1, 2, 4], [1, 2, 4, 8, 16]])
def test_one_group_where_a_wave_is_one_group(npix, dts):
    with _plan(npix, [1]) as one, _plan(npix, dts) as many:
        group = 32 * (one.info().iu_max + 1) * npix * 8
        more = _estimate(many, 32) - _estimate(one, 32)
        assert more < group / 4 + 2 ** 20  # series of the other widths, lists and records: under a megabyte here
        # a wave of 256 images holds 256 transformed ones at most
        assert _estimate(many, 256) <= _estimate(one, 256) + group / 4 + 2 ** 20


@pytest.mark.parametrize("npix,dts", [(256, [1]), (1024, [1, 2]), (2048, [1, 2, 4, 8])])
def test_clipped_noise_partials_lie_in_the_cell_buffer(npix, dts):
    with _plan(npix, dts) as plain, _plan(npix, dts, rf.RF_NOISE_CLIPPED) as clipped:
        # beside a window an image: what the partials, 16 bytes a row pair or a
        # row of an image, take beyond the cell sums of two to four groups
        partials = 64 * npix // 2 * 16 * (2 if 8 in dts else 1) * (npix // 1024 if npix > 1024 else 1)
        cells = plain.info().n_cells * 32 * 8
        more = _estimate(clipped, 64) - _estimate(plain, 64) - 64 * 8
        assert partials - 4 * cells <= more <= partials - 2 * cells
