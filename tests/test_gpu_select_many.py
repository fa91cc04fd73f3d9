"""Persistent blocks that take many units, some by the whole-unit selection
(flat frames: more equal values than the candidate lists hold; frames far below
the window) and some by the ranked candidates, in no order: every form of the
median.  Reference: the CPU oracle, bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1903_06838_gb300 import pd, synth
from tests._cases import sort_hits

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = {  # the units of a block of 304: more than six
    "banks": (dict(n_modules=1, rows=64, cols=128, unit_rows=64, unit_cols=64), 1000),
    "rows": (dict(n_modules=1, rows=32, cols=128, unit_rows=1, unit_cols=128), 500),
    "blocks": (dict(n_modules=1, rows=24, cols=90, unit_rows=12, unit_cols=45), 800),
}


@pytest.mark.parametrize("tuning", [dict(kernels=1), dict(kernels=2), dict(kernels=3),
                                    dict(two_pass=0), dict(mixed=True)],
                         ids=["lean", "earlier", "queue", "one_kernel", "mixed"])
@pytest.mark.parametrize("shape", list(SHAPES))
def test_selections_in_any_order(shape, tuning):
    geometry, n = SHAPES[shape]
    det = synth.Detector(occupancy=0.01, **geometry)
    ped, gain = synth.maps(det)
    ped = np.round(ped)
    raw, _ = synth.frames(det, ped, gain, 0, n, truth=False)
    rng = np.random.default_rng(3)
    raw = raw.reshape(n, 1, det.rows, det.cols)
    how = rng.integers(0, 3, n)
    raw[how == 1] = ped.astype(np.uint16)[None]               # flat
    raw[how == 2] = raw[how == 2] - np.uint16(900)            # below every window
    raw[how == 2, :, ::7, ::9] += np.uint16(900 + 300)        # and photons
    thr = det.thresholds()
    ctx = pd.pd_create(det.geometry(), ped, gain, thr)
    mixed = tuning.get("mixed")
    pd.pd_set_tuning(ctx, **{k: v for k, v in tuning.items() if k != "mixed"})
    dev = pd.frames_to_device(raw)
    out = pd.Outputs(ctx, n, raw.size // 4 + 64, cm=True)
    if mixed:
        batch = pd.pd_batch_create(1)
        pd.pd_batch_set_mixed(batch, True)
        pd.pd_batch_process(batch, [(ctx, dev.data_ptr(), n, 0, out)])
    else:
        pd.pd_process(ctx, dev.data_ptr(), n, 0, **out.ptrs())
    torch.cuda.synchronize()
    ref = oracle.process(oracle.geometry(**det.geometry()), oracle.thresholds(**thr), ped, gain, raw,
                         hit_capacity=raw.size // 4 + 64)
    assert out.cm.cpu().numpy().tobytes() == ref.cm.reshape(n, -1).tobytes()
    hits, nh = out.hits_host()
    assert nh == ref.n_hits
    assert sort_hits(hits).tobytes() == sort_hits(ref.hits).tobytes()
