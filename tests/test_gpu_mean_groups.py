"""The fused rows and columns of the stacked mean for every number of column
pairs a lane holds: the widest module of each, and one column pair past the
narrower one's.  Reference: the CPU oracle, bit for bit."""
from __future__ import annotations

import pytest

import oracle
from paper_1903_06838_gb300 import pd, synth
from tests._cases import sort_hits

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("groups", range(1, 17))
def test_every_group_count(groups):
    for cols in {min(64 * groups, 1000), 64 * (groups - 1) + 2}:
        det = synth.Detector(n_modules=2, rows=19, cols=cols, unit_rows=19, unit_cols=cols,
                             occupancy=0.02, seed=groups)
        ped, gain = synth.maps(det)
        raw, _ = synth.frames(det, ped, gain, 0, 2, truth=False)
        geom = dict(det.geometry(), cm_mode=pd.PD_CM_MEAN_STACKED)
        thr = det.thresholds()
        ctx = pd.pd_create(geom, ped, gain, thr)
        out = pd.process(ctx, pd.frames_to_device(raw), hit_capacity=raw.size, corrected=True,
                         cm=True)
        torch.cuda.synchronize()
        ref = oracle.process(oracle.geometry(**geom), oracle.thresholds(**thr), ped, gain, raw,
                             want_corrected=True, hit_capacity=raw.size)
        hits, n = out.hits_host()
        assert n == ref.n_hits
        assert sort_hits(hits).tobytes() == sort_hits(ref.hits).tobytes()
        assert out.cm.cpu().numpy().tobytes() == ref.cm.reshape(2, -1).tobytes()
        assert out.corrected.cpu().numpy().tobytes() == ref.corrected.reshape(2, -1).tobytes()
