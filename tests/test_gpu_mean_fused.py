"""The mean common mode's one-pass unit sums and its fused row and column
stages, and the lean stencil's stacked and auto-ranging instances, at the
sizes where they change: the lanes' column-pair counts, more and fewer rows
than warps, one-row and one-column-pair units, widths the fused stages leave
to the separate kernels, pedestals whose binary places rule out the one-pass
sums, cuts that select nothing or everything; against the CPU oracle, bit for
bit, with both kernel pairs."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1903_06838_gb300 import pd, synth
from tests._cases import sort_hits

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

#        modules, rows, cols, unit_rows, unit_cols
SIZES = {
    "one_pair": (2, 9, 2, 9, 2),
    "lanes_less_one": (1, 8, 62, 8, 62),
    "lanes_full": (1, 7, 64, 1, 64),
    "three_pairs_edge": (2, 33, 192, 33, 64),
    "three_pairs_past": (1, 1, 194, 1, 194),
    "six_pairs_edge": (1, 40, 384, 20, 192),
    "seven_pairs_edge": (1, 17, 448, 17, 224),
    "twelve_pairs": (1, 16, 450, 8, 50),
    "twelve_pairs_edge": (1, 5, 768, 5, 384),
    "sixteen_pairs": (1, 12, 770, 12, 10),
    "widest_fused": (1, 3, 1000, 3, 500),
    "past_fused": (1, 3, 1002, 3, 334),
    "odd_columns": (1, 11, 45, 11, 15),
    "odd_units": (1, 10, 90, 10, 45),
}


def _check(det, geom, thr, ped, gain, raw, kernels=0, **gains):
    n = raw.shape[0]
    ctx = pd.pd_create(geom, ped, gain, thr, **gains)
    if kernels:
        pd.pd_set_tuning(ctx, kernels=kernels)
    cap = n * det.pixels_per_frame
    out = pd.process(ctx, pd.frames_to_device(raw), hit_capacity=cap, corrected=True, cm=True)
    torch.cuda.synchronize()
    ref = oracle.process(oracle.geometry(**geom), oracle.thresholds(**thr), ped, gain, raw,
                         want_corrected=True, hit_capacity=cap, **gains)
    hits, nh = out.hits_host()
    assert nh == ref.n_hits
    assert sort_hits(hits).tobytes() == sort_hits(ref.hits).tobytes()
    assert out.cm.cpu().numpy().tobytes() == ref.cm.reshape(n, -1).tobytes()
    assert out.corrected.cpu().numpy().tobytes() == ref.corrected.reshape(n, -1).tobytes()
    for got, exp in zip(pd.pd_get_summary(ctx), (ref.count_map, ref.hist_pix, ref.hist_hit)):
        np.testing.assert_array_equal(got, exp)


def _data(size, n=2, seed=5):
    m, r, c, ur, uc = SIZES[size]
    det = synth.Detector(n_modules=m, rows=r, cols=c, unit_rows=ur, unit_cols=uc,
                         occupancy=0.03, seed=seed)
    ped, gain = synth.maps(det)
    raw, _ = synth.frames(det, ped, gain, 0, n, truth=False)
    return det, ped, gain, raw


@pytest.mark.parametrize("kernels", [1, 2])
@pytest.mark.parametrize("mode", [pd.PD_CM_MEAN, pd.PD_CM_MEAN_STACKED])
@pytest.mark.parametrize("size", list(SIZES))
def test_sizes(size, mode, kernels):
    det, ped, gain, raw = _data(size)
    _check(det, dict(det.geometry(), cm_mode=mode), det.thresholds(), ped, gain, raw, kernels)


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("mode", [pd.PD_CM_MEAN, pd.PD_CM_MEAN_STACKED])
@pytest.mark.parametrize("kind", ["whole", "zero", "negative", "fine", "huge", "cut_low",
                                  "cut_high", "masked"])
def test_pedestals_and_cuts(kind, mode, order):
    det, ped, gain, raw = _data("six_pairs_edge")
    thr = det.thresholds()
    if kind == "whole":      # no binary places: the coarsest one-pass grid
        ped = np.round(ped)
    elif kind == "zero":     # d = raw
        ped = np.zeros_like(ped)
    elif kind == "negative":
        ped = -ped
    elif kind == "fine":     # 24 places and more: the two-pass sums
        ped[0, 3, 5:9] = np.float32(3.0e-7)
        ped[0, 4, 7] = np.float32(1e-30)
        raw[:, 0, 3, 5:9] = [1, 0, 2, 0]
        raw[:, 0, 4, 7] = 0
    elif kind == "huge":     # d not exact in binary32, values beyond 2^26 places
        ped[0, 2, :40] = np.float32(3.0e7)
        ped[0, 9, 3] = np.float32(-2.5e9)
    elif kind == "cut_low":
        thr.update(cm_cut_adu=-1000.0, cm_cut_kev=-40.0)
    elif kind == "cut_high":
        thr.update(cm_cut_adu=70000.0, cm_cut_kev=3000.0)
    elif kind == "masked":
        gain[0, :, 17] = 0.0
        gain[0, 21] = -1.0
    _check(det, dict(det.geometry(), cm_mode=mode, cm_after_gain=order), thr, ped, gain, raw)


@pytest.mark.parametrize("kernels", [1, 2])
@pytest.mark.parametrize("shift", [10, 11, 12, 14, 15])
@pytest.mark.parametrize("name", ["banks", "blocks", "rows"])
def test_auto_ranging_raw_cap(name, shift, kernels):
    # a stage field from bit 10 or 11 leaves the bank median's raw cap (about
    # 1900 here) above the stage step, where it does not apply
    shape = {"banks": (2, 70, 128, 70, 64), "blocks": (1, 140, 128, 70, 64),
             "rows": (1, 40, 128, 1, 128)}[name]
    m, r, c, ur, uc = shape
    det = synth.Detector(n_modules=m, rows=r, cols=c, unit_rows=ur, unit_cols=uc, occupancy=0.02,
                         ped_mean=500.0 if shift < 12 else 1500.0, ped_sigma=20.0)
    ped, gain = synth.multigain_maps(det, 2, (1.0, 0.1), (0.0, -200.0))
    raw, _ = synth.multigain_frames(det, ped, gain, 0, 2, gain_shift=shift, blob_kev=200.0,
                                    bad_frac=1e-3)
    for mode in (pd.PD_CM_MEDIAN, pd.PD_CM_NONE):
        _check(det, dict(det.geometry(), cm_mode=mode), det.thresholds(), ped, gain, raw, kernels,
               n_gains=2, gain_shift=shift)
