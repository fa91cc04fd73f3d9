"""The one-kernel chain on modules so narrow that their own threads are less
than a warp for each of their two banks: columns 4 to 64, few and many rows.
Reference: the CPU oracle, bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1903_06838_gb300 import pd, synth
from tests._cases import sort_hits

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cols", [4, 8, 24, 40, 52, 64])
@pytest.mark.parametrize("rows", [3, 150])
@pytest.mark.parametrize("banks", [1, 2])
def test_narrow_modules(cols, rows, banks):
    det = synth.Detector(n_modules=3, rows=rows, cols=cols, unit_rows=rows,
                         unit_cols=cols // banks, occupancy=0.03)
    ped, gain = synth.maps(det)
    raw, _ = synth.frames(det, ped, gain, 0, 5, truth=False)
    ctx = pd.pd_create(det.geometry(), ped, gain, det.thresholds())
    pd.pd_set_tuning(ctx, two_pass=0)
    if pd.pd_get_tuning(ctx)["two_pass"]:
        pytest.skip("the one-kernel form does not take this geometry")
    out = pd.process(ctx, pd.frames_to_device(raw), hit_capacity=raw.size, corrected=True, cm=True)
    torch.cuda.synchronize()
    ref = oracle.process(oracle.geometry(**det.geometry()), oracle.thresholds(**det.thresholds()),
                         ped, gain, raw, want_corrected=True, hit_capacity=raw.size)
    hits, n = out.hits_host()
    assert n == ref.n_hits > 0
    assert sort_hits(hits).tobytes() == sort_hits(ref.hits).tobytes()
    assert out.cm.cpu().numpy().tobytes() == ref.cm.reshape(len(raw), -1).tobytes()
    assert out.corrected.cpu().numpy().tobytes() == ref.corrected.tobytes()
    for got, exp in zip(pd.pd_get_summary(ctx), (ref.count_map, ref.hist_pix, ref.hist_hit)):
        np.testing.assert_array_equal(got, exp)
