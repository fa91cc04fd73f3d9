"""Calls of few tiles take shorter bands: one, two and many frames of small
modules through each band stencil (four-pixel chunks with and without staged
raw rows, single pixels, the matched filters), heights that divide the module
and that leave a ragged last band, against the CPU oracle, bit for bit; and an
explicit height is kept."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1903_06838_gb300 import filters, pd, synth
from tests._cases import sort_hits

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = {
    "staged": dict(rows=97, cols=64, unit_rows=1, unit_cols=64),
    "chunks": dict(rows=185, cols=388, unit_rows=185, unit_cols=194),
    "one_row_lane": dict(rows=24, cols=2044, unit_rows=24, unit_cols=511),
    "pixels": dict(rows=131, cols=75, unit_rows=131, unit_cols=25),
    "single_row": dict(rows=1, cols=384, unit_rows=1, unit_cols=384),
}


@pytest.mark.parametrize("matched", [False, True])
@pytest.mark.parametrize("frames", [1, 2, 40])
@pytest.mark.parametrize("shape", list(SHAPES))
def test_small_calls(shape, frames, matched):
    det = synth.Detector(n_modules=2, occupancy=0.03, **SHAPES[shape])
    ped, gain = synth.maps(det)
    raw, _ = synth.frames(det, ped, gain, 0, frames, truth=False)
    geom, thr = det.geometry(), det.thresholds()
    bank = filters.example_bank() if matched else None
    okw = dict(filters=oracle.filters(**bank)) if matched else {}
    ref = oracle.process(oracle.geometry(**geom), oracle.thresholds(**thr), ped, gain, raw,
                         want_corrected=True, **okw)
    for band_rows in (0, 5):
        ctx = pd.pd_create(geom, ped, gain, thr)
        if matched:
            pd.pd_set_filter_bank(ctx, **bank)
        if band_rows:
            pd.pd_set_tuning(ctx, band_rows=band_rows)
        out = pd.process(ctx, pd.frames_to_device(raw), corrected=True, cm=True)
        torch.cuda.synchronize()
        hits, n = out.hits_host()
        assert n == ref.n_hits
        assert sort_hits(hits).tobytes() == sort_hits(ref.hits).tobytes()
        assert out.corrected.cpu().numpy().ravel().tobytes() == ref.corrected.ravel().tobytes()
        cmap, hp, hh = pd.pd_get_summary(ctx)
        assert np.array_equal(cmap, ref.count_map)
        assert np.array_equal(hp, ref.hist_pix) and np.array_equal(hh, ref.hist_hit)
