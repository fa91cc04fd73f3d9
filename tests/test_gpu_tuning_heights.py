"""Band heights of the stacked mean and of auto-ranging words: their contexts
ran the band stencil, which holds taller bands than the lean one, and every
height it takes stays accepted: the lean stencil then takes the tallest it
holds.  Past what either holds, the call is refused and the heights stay.
Results against the CPU oracle."""
from __future__ import annotations

import pytest

import oracle
from paper_1903_06838_gb300 import pd, synth
from tests._cases import sort_hits

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (columns, rows, a height the band stencil holds and the lean one does not)
SIZES = {"388": (388, 120, 100), "2048": (2048, 24, 18)}


def _context(size, kind):
    cols, rows, _ = SIZES[size]
    det = synth.Detector(n_modules=1, rows=rows, cols=cols, unit_rows=rows, unit_cols=cols // 2,
                         occupancy=0.02)
    thr = det.thresholds()
    if kind == "stacked":
        geom, kw = dict(det.geometry(), cm_mode=pd.PD_CM_MEAN_STACKED), {}
        ped, gain = synth.maps(det)
        raw, _ = synth.frames(det, ped, gain, 0, 2, truth=False)
    else:
        geom, kw = det.geometry(), dict(n_gains=2, gain_shift=14)
        ped, gain = synth.multigain_maps(det, 2, (1.0, 0.1), (0.0, -200.0))
        raw, _ = synth.multigain_frames(det, ped, gain, 0, 2, gain_shift=14, blob_kev=200.0,
                                        bad_frac=1e-3)
    ref = oracle.process(oracle.geometry(**geom), oracle.thresholds(**thr), ped, gain, raw,
                         hit_capacity=raw.size, **kw)
    return pd.pd_create(geom, ped, gain, thr, **kw), raw, ref


@pytest.mark.parametrize("kind", ["stacked", "auto_ranging"])
@pytest.mark.parametrize("size", list(SIZES))
def test_band_stencils_heights_stay_accepted(size, kind):
    cols, rows, height = SIZES[size]
    ctx, raw, ref = _context(size, kind)
    pd.pd_set_tuning(ctx, band_rows=height)
    assert pd.pd_get_tuning(ctx)["kernels"] == 1
    assert 0 < pd.pd_get_tuning(ctx)["band_rows"] < height
    for kernels in (1, 2):
        pd.pd_set_tuning(ctx, kernels=kernels)
        out = pd.process(ctx, pd.frames_to_device(raw), hit_capacity=raw.size)
        torch.cuda.synchronize()
        hits, n = out.hits_host()
        assert n == ref.n_hits > 0
        assert sort_hits(hits).tobytes() == sort_hits(ref.hits).tobytes()
    assert pd.pd_get_tuning(ctx)["band_rows"] == height  # of the band stencil (kernels 2)


@pytest.mark.parametrize("mode", [pd.PD_CM_MEDIAN, pd.PD_CM_MEAN_STACKED])
def test_refused_height_changes_no_height(mode):
    det = synth.Detector(n_modules=1, rows=600, cols=512, unit_rows=600, unit_cols=256)
    ped, gain = synth.maps(det)
    ctx = pd.pd_create(dict(det.geometry(), cm_mode=mode), ped, gain, det.thresholds())
    pd.pd_set_tuning(ctx, band_rows=20)
    with pytest.raises(pd.PdError) as e:
        pd.pd_set_tuning(ctx, band_rows=600)
    assert e.value.code == pd.PD_EINVAL
    for kernels in (1, 2):
        pd.pd_set_tuning(ctx, kernels=kernels)
        assert pd.pd_get_tuning(ctx)["band_rows"] == 20
