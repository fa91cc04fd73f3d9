"""Energies far outside the pixel histogram go to its end bins: distances of up
to 2^50 bins on either side, past the range in which the bin is found by a
magic addition, in every stencil.  Reference: the CPU oracle."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1903_06838_gb300 import filters, pd

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROWS, COLS = 16, 72


@pytest.mark.parametrize("cols", [COLS, COLS - 1])  # chunks of four, single pixels
@pytest.mark.parametrize("how", ["lean", "band", "matched", "stacked", "auto_ranging"])
def test_end_bins(how, cols):
    rng = np.random.default_rng(2)
    ped = np.full((1, ROWS, cols), 20000.0, np.float32)
    gain = np.exp2(-rng.uniform(0.0, 32.0, (1, ROWS, cols))).astype(np.float32)
    raw = (20000 + rng.integers(-15000, 15000, (2, 1, ROWS, cols))).astype(np.uint16)
    geom = dict(n_modules=1, rows=ROWS, cols=cols, unit_rows=ROWS, unit_cols=cols,
                cm_mode=pd.PD_CM_MEAN_STACKED if how == "stacked" else pd.PD_CM_NONE)
    thr = dict(cm_cut_adu=100.0, zero_thr_kev=3e38, seed_thr_kev=3e38, photon_kev=8.0,
               hist_lo_kev=-4.0, hist_bin_kev=0.05, hist_bins=1296)
    kw = {}
    if how == "auto_ranging":
        kw = dict(n_gains=2, gain_shift=15)
        ped, gain = np.stack([ped, ped]), np.stack([gain, gain])
    ctx = pd.pd_create(geom, ped, gain, thr, **kw)
    okw = dict(kw)
    if how == "matched":
        bank = filters.example_bank()
        pd.pd_set_filter_bank(ctx, **bank)
        okw["filters"] = oracle.filters(**bank)
    pd.pd_set_tuning(ctx, kernels=2 if how == "band" else 1)
    pd.process(ctx, pd.frames_to_device(raw))
    ref = oracle.process(oracle.geometry(**geom), oracle.thresholds(**thr), ped, gain, raw, **okw)
    assert ref.hist_pix[0] > 100 and ref.hist_pix[-1] > 100
    np.testing.assert_array_equal(pd.pd_get_summary(ctx)[1], ref.hist_pix)
