"""The noise's sums over the cells of a column add in short chains.

One cell of power 1 and 483 others of just under half its last place, all in one
column: a cell added to a sum that holds the bright one is lost.  A chain takes
every 32nd cell, so the 15 after the bright one are lost, 15 x 2^-24 of the
power and half that of sigma (4.5e-7); five additions of a tree round by 2^-24
each (1.5e-7 of sigma), the record by 6e-8: 8e-7 is asked for.  Chains of every
8th cell lose 60 (1.8e-6).
"""

import numpy as np
import pytest

import oracle
import paper_1802_03084_gb300 as rf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npix,dts", [(1024, [1]), (1024, [1, 2, 4]), (1024, [1, 2, 4, 8, 16]), (2048, [1, 2, 16]),
                                      (4096, [1, 4])])
def test_faint_cells_beside_a_bright_one(npix, dts):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    # two north-south lines 37 cells apart: spacings 22 and 1, so 484 baselines in 484 cells of column 37
    k, nint = 22, 35
    ant = np.zeros((2 * k, 3))
    ant[:k, 1] = 10.0 * k * np.arange(k)
    ant[k:, 1] = 10.0 * np.arange(k)
    ant[k:, 0] = 370.0
    i, j = np.triu_indices(2 * k, k=1)
    across = (i < k) & (j >= k)
    faint = np.float32(np.sqrt(0.99 * 2.0 ** -24))
    vis = np.zeros((nint, len(i), 1, 1), dtype=np.complex64)
    vis[:, across] = faint
    vis[:, across & (i == 0) & (j == k)] = 1.0  # v = 0: the column's first cell
    power = float(1.0 + (across.sum() - 1) * float(faint) ** 2)
    with rf.Plan(ant, np.array([oracle.C_LIGHT]), 1e-3, npix, 0.1 / npix, np.array([0.0]), dts, 5.0, npol=1,
                 max_nint=nint) as gp:
        stats = gp.search_stats(vis)[1]
    assert set(stats["dt_idx"]) == set(range(len(dts)))
    # sum of |G|^2 over the full plane, over 4 W^2; the samples of a width add in FP32 without rounding up to 16
    sigma = np.sqrt(2.0 * power) / (2.0 * len(i))
    assert np.all(stats["weight"] == len(i) * np.array(dts)[stats["dt_idx"]])
    assert np.max(np.abs(stats["sigma"] / sigma - 1.0)) < 8e-7
