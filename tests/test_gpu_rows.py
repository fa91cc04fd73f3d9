"""The coded median of one-row units at the sizes and values where it changes:
lanes with one to four chunks, full and not, rows whose values share one code,
lie below the window, sit at the cut or miss the minimum count, several units
per row, more units than persistent warps, auto-ranging words with the stage
field above and below the raw cap; the common mode against the CPU oracle, bit
for bit, with both kernel pairs."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1903_06838_gb300 import pd, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _cm(det, thr, ped, gain, raw, kernels, **gains):
    geom = det.geometry()
    ctx = pd.pd_create(geom, ped, gain, thr, **gains)
    pd.pd_set_tuning(ctx, kernels=kernels)
    out = pd.process(ctx, pd.frames_to_device(raw), cm=True)
    torch.cuda.synchronize()
    ref = oracle.process(oracle.geometry(**geom), oracle.thresholds(**thr), ped, gain, raw,
                         hit_capacity=1 << 20, **gains)
    assert int(out.n_hits.item()) == ref.n_hits
    return out.cm.cpu().numpy().ravel(), ref.cm.ravel()


def _det(rows, unit_cols, per_row=1, **kw):
    return synth.Detector(n_modules=1, rows=rows, cols=unit_cols * per_row, unit_rows=1,
                          unit_cols=unit_cols, **kw)


@pytest.mark.parametrize("kernels", [1, 2])
@pytest.mark.parametrize("unit_cols", [4, 8, 44, 124, 128, 132, 256, 260, 380, 384, 388, 508, 512])
def test_unit_sizes(unit_cols, kernels):
    det = _det(37, unit_cols, 2 if unit_cols < 300 else 1, occupancy=0.05)
    ped, gain = synth.maps(det)
    raw, _ = synth.frames(det, ped, gain, 0, 3, truth=False)
    got, ref = _cm(det, det.thresholds(), ped, gain, raw, kernels)
    assert got.tobytes() == ref.tobytes()


@pytest.mark.parametrize("kernels", [1, 2])
@pytest.mark.parametrize("kev", [6.0, 12.0, 40.0])
def test_values(kev, kernels):
    det = _det(16, 384, photon_kev=kev, occupancy=0.02)
    ped, gain = synth.maps(det)
    raw, _ = synth.frames(det, ped, gain, 0, 2, truth=False)
    p0 = np.round(ped).astype(np.int64)
    cut = int(kev * 25)
    raw[:, 0, 0] = (p0[0, 0] + 3).astype(np.uint16)       # values within one ADU
    ped[0, 1] = 1500.0
    raw[:, 0, 1] = 1504                                   # one value
    ped[0, 2] = 1500.0
    raw[:, 0, 2, ::2], raw[:, 0, 2, 1::2] = 1500, 1501    # two values, even count
    raw[:, 0, 3] = 0                                      # below the window
    raw[:, 0, 4] = 65535                                  # nothing below the cut
    raw[:, 0, 5, 19:] = 65535                             # one short of the minimum
    raw[:, 0, 6, 20:] = 65535                             # the minimum (ceil(sqrt(384)))
    ped[0, 7] = 1500.0
    raw[:, 0, 7] = 1500 + cut                             # at the cut: excluded
    raw[:, 0, 7, :40] = 1500 + cut - 1
    raw[0, 0, 8] = np.arange(384) + 1300                  # a ramp
    raw[1, 0, 8] = 1500 + (np.arange(384) % 2) * 150      # two far groups
    ped[0, 9] = 1500.0 + np.arange(384, dtype=np.float32) * np.float32(2.0 ** -13)
    raw[:, 0, 9] = 1500                                   # 384 values in one code
    got, ref = _cm(det, det.thresholds(), ped, gain, raw, kernels)
    assert got.tobytes() == ref.tobytes()


def test_more_units_than_warps():
    det = _det(352, 128, 3, occupancy=0.02)
    ped, gain = synth.maps(det)
    raw, _ = synth.frames(det, ped, gain, 0, 11, truth=False)
    got, ref = _cm(det, det.thresholds(), ped, gain, raw, 1)
    assert got.tobytes() == ref.tobytes()


@pytest.mark.parametrize("ped_mean", [300.0, 900.0, 3000.0, 9000.0])
def test_pedestal_ranges(ped_mean):
    det = _det(20, 384, ped_mean=ped_mean, ped_sigma=ped_mean / 8, occupancy=0.02)
    ped, gain = synth.maps(det)
    raw, _ = synth.frames(det, ped, gain, 0, 2, truth=False)
    got, ref = _cm(det, det.thresholds(), ped, gain, raw, 1)
    assert got.tobytes() == ref.tobytes()


@pytest.mark.parametrize("shift", [10, 11, 12, 14])
def test_auto_ranging_words(shift):
    det = _det(24, 256, occupancy=0.02, ped_mean=500.0 if shift < 12 else 1500.0, ped_sigma=20.0)
    ped, gain = synth.multigain_maps(det, 3, (1.0, 0.1, 0.01), (0.0, -100.0, -200.0))
    raw, _ = synth.multigain_frames(det, ped, gain, 0, 2, gain_shift=shift, blob_kev=300.0,
                                    bad_frac=1e-3)
    got, ref = _cm(det, det.thresholds(), ped, gain, raw, 1, n_gains=3, gain_shift=shift)
    assert got.tobytes() == ref.tobytes()
