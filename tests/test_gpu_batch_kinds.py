"""One persistent common-mode launch over units of every kind: a block takes
large units whose median lies below the window or in a bin of too many values
(the whole-unit selection), then units of the generic and of the row kind, and
the other way round.  Reference: the CPU oracle, bit for bit."""
from __future__ import annotations

import itertools

import numpy as np
import pytest

import oracle
from paper_1903_06838_gb300 import pd, synth
from tests._cases import sort_hits

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# name: detector, cut (ADU), frames; more than 304 tasks in all, so that a block
# takes several
KINDS = {
    "below_window": (dict(n_modules=3, rows=31, cols=768, unit_rows=31, unit_cols=384), 70000.0, 30),
    "flat": (dict(n_modules=2, rows=56, cols=768, unit_rows=56, unit_cols=384, noise_sigma=0.0),
             200.0, 30),
    "odd_large": (dict(n_modules=2, rows=70, cols=75, unit_rows=70, unit_cols=75), 70000.0, 60),
    "generic": (dict(n_modules=2, rows=12, cols=137, unit_rows=12, unit_cols=137), 200.0, 200),
    "small_generic": (dict(n_modules=1, rows=3, cols=64, unit_rows=3, unit_cols=4), 137.3, 30),
    "rows": (dict(n_modules=1, rows=352, cols=384, unit_rows=1, unit_cols=384), 200.0, 20),
}
ORDERS = list(itertools.permutations(("below_window", "generic", "rows"))) + [
    ("flat", "generic", "small_generic"), ("odd_large", "small_generic", "generic"),
    ("small_generic", "flat", "generic", "odd_large", "rows"),
    # (a kernel of its own: large units of column pairs, and rows)
    ("below_window", "rows"), ("flat", "rows", "below_window"), ("flat", "flat", "below_window")]


@pytest.mark.parametrize("order", ORDERS, ids=lambda o: "+".join(o))
def test_kinds_in_one_launch(order):
    items, refs, keep = [], [], []
    for name in order:
        shape, cut, frames = KINDS[name]
        det = synth.Detector(occupancy=0.02, **shape)
        ped, gain = synth.maps(det)
        if name == "flat":
            ped = np.round(ped)
        raw, _ = synth.frames(det, ped, gain, 0, frames, truth=False)
        thr = dict(det.thresholds(), cm_cut_adu=cut)
        ctx = pd.pd_create(det.geometry(), ped, gain, thr)
        dev = pd.frames_to_device(raw)
        out = pd.Outputs(ctx, frames, raw.size // 4 + 64, cm=True)
        items.append((ctx, dev.data_ptr(), frames, 0, out))
        keep.append(dev)
        refs.append(oracle.process(oracle.geometry(**det.geometry()), oracle.thresholds(**thr), ped,
                                   gain, raw, hit_capacity=raw.size // 4 + 64))
    batch = pd.pd_batch_create(len(items))
    pd.pd_batch_set_mixed(batch, True)
    pd.pd_batch_process(batch, items)
    torch.cuda.synchronize()
    for name, (ctx, _, frames, _, out), ref in zip(order, items, refs):
        assert out.cm.cpu().numpy().tobytes() == ref.cm.reshape(frames, -1).tobytes(), name
        hits, n = out.hits_host()
        assert n == ref.n_hits
        assert sort_hits(hits).tobytes() == sort_hits(ref.hits).tobytes()
