"""The paper's order through the band stencil and beside it: the band height is
reported, set and tuned as for the other contexts, and the contexts that the
band stencil does not take (rows wider than its block; energies so large that
their difference could overflow) keep the tile stencil.  Reference: the CPU
oracle, bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1903_06838_gb300 import pd, synth
from tests._cases import sort_hits

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MODES = {"median": pd.PD_CM_MEDIAN, "mean": pd.PD_CM_MEAN, "stacked": pd.PD_CM_MEAN_STACKED}
SHAPES = {
    "pixels": dict(n_modules=2, rows=61, cols=75, unit_rows=61, unit_cols=25),
    "chunks": dict(n_modules=2, rows=61, cols=128, unit_rows=61, unit_cols=64),
    "wide_odd": dict(n_modules=1, rows=21, cols=515, unit_rows=21, unit_cols=103),
}


def _case(shape, mode, scale=0, n=3):
    """scale: gains and energies in units of 2^scale keV (exact)."""
    det = synth.Detector(occupancy=0.03, **SHAPES[shape])
    ped, gain = synth.maps(det)
    gain.reshape(-1)[::53] = 0.0
    raw, _ = synth.frames(det, ped, gain, 0, n, truth=False)
    gain = np.ldexp(gain, -scale).astype(np.float32)
    geom = dict(det.geometry(), cm_mode=MODES[mode], cm_after_gain=1)
    thr = dict(det.thresholds())
    thr.update(hist_lo_kev=-4.0, hist_bin_kev=0.0625, hist_bins=1200, cm_cut_kev=thr["photon_kev"])
    for k in ("zero_thr_kev", "seed_thr_kev", "photon_kev", "hist_lo_kev", "hist_bin_kev",
              "cm_cut_kev"):
        thr[k] = float(np.ldexp(thr[k], scale))
    ref = oracle.process(oracle.geometry(**geom), oracle.thresholds(**thr), ped, gain, raw,
                         want_corrected=True, hit_capacity=raw.size)
    assert ref.n_hits > 0
    return pd.pd_create(geom, ped, gain, thr), raw, ref


def _compare(ctx, raw, ref):
    n = len(raw)
    pd.pd_reset_summary(ctx)
    out = pd.process(ctx, pd.frames_to_device(raw), hit_capacity=raw.size, corrected=True, cm=True)
    torch.cuda.synchronize()
    hits, nh = out.hits_host()
    assert nh == ref.n_hits
    assert sort_hits(hits).tobytes() == sort_hits(ref.hits).tobytes()
    assert out.cm.cpu().numpy().tobytes() == ref.cm.reshape(n, -1).tobytes()
    assert out.corrected.cpu().numpy().tobytes() == ref.corrected.reshape(n, -1).tobytes()
    for got, exp in zip(pd.pd_get_summary(ctx), (ref.count_map, ref.hist_pix, ref.hist_hit)):
        np.testing.assert_array_equal(got, exp)


@pytest.mark.parametrize("mode", list(MODES))
@pytest.mark.parametrize("shape", ["pixels", "chunks"])
def test_band_height_reaches_the_stencil(shape, mode):
    ctx, raw, ref = _case(shape, mode)
    rows = SHAPES[shape]["rows"]
    assert 0 < pd.pd_get_tuning(ctx)["band_rows"] <= rows
    for height in (1, 7, rows):
        pd.pd_set_tuning(ctx, band_rows=height)
        assert pd.pd_get_tuning(ctx)["band_rows"] == height
        _compare(ctx, raw, ref)
    pd.pd_set_tuning(ctx, band_rows=10 ** 6)
    assert pd.pd_get_tuning(ctx)["band_rows"] == rows
    dev = pd.frames_to_device(raw)
    best, _ = pd.pd_autotune(ctx, dev.data_ptr(), len(raw))
    assert best["band_rows"] > 0
    _compare(ctx, raw, ref)


def test_height_past_shared_memory_takes_the_tallest():
    # 515 rows of 512 columns do not fit an SM
    det = synth.Detector(n_modules=1, rows=515, cols=512, unit_rows=515, unit_cols=512)
    ped, gain = synth.maps(det)
    geom = dict(det.geometry(), cm_mode=pd.PD_CM_MEAN, cm_after_gain=1)
    ctx = pd.pd_create(geom, ped, gain, det.thresholds())
    pd.pd_set_tuning(ctx, band_rows=515)
    got = pd.pd_get_tuning(ctx)["band_rows"]
    assert 0 < got < 515 and (got + 3) * 512 * 4 < 200 * 1024 < (got + 30) * 512 * 4
    raw, _ = synth.frames(det, ped, gain, 0, 1, truth=False)
    ref = oracle.process(oracle.geometry(**geom), oracle.thresholds(**det.thresholds()), ped, gain,
                         raw, want_corrected=True, hit_capacity=raw.size)
    _compare(ctx, raw, ref)


@pytest.mark.parametrize("mode", list(MODES))
@pytest.mark.parametrize("shape,scale,bands", [
    ("chunks", 111, True), ("chunks", 112, False), ("pixels", 111, True), ("pixels", 112, False),
    ("wide_odd", 0, False)])
def test_both_sides_of_the_rule(shape, scale, bands, mode):
    # (65536 + pedestal) / gain is 0.8e37 at 2^111 and 1.6e37 at 2^112, the
    # rule's line 1e37
    ctx, raw, ref = _case(shape, mode, scale)
    assert (pd.pd_get_tuning(ctx)["band_rows"] > 0) == bands
    _compare(ctx, raw, ref)
