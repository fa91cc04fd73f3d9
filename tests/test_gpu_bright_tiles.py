"""Tiles with many seed candidates.

A tile of the lean stencil with more candidates than threads tests them all
before it sums any.  Neighbours without an energy (NaN: a gain so small that its
inverse is infinite, on a pixel whose signal is exactly 0) count as no signal
there as they do elsewhere.  Reference: the CPU oracle, bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1903_06838_gb300 import pd
from tests._cases import sort_hits

torch = pytest.importorskip("torch")

ROWS, COLS = 61, 388
BAND = 20       # rows of a tile: not the default height, which calls of one frame cut
GEOM = dict(n_modules=1, rows=ROWS, cols=COLS, unit_rows=ROWS, unit_cols=COLS // 2)
THR = dict(cm_cut_adu=200.0, zero_thr_kev=0.8, seed_thr_kev=0.8, photon_kev=8.0)
THREADS = 512  # the most a tile's block has
LIST = 4096    # candidates a tile's list holds

# neighbours (row, column) of a seed that have no energy
NEIGHBOURS = {
    "before": [(-1, -1), (-1, 0), (-1, 1), (0, -1)],
    "after": [(0, 1), (1, -1), (1, 0), (1, 1)],
    "all": [(i, j) for i in (-1, 0, 1) for j in (-1, 0, 1) if i or j],
    "one_each": [(-1, 0), (1, 0)],
}


def _case(which):
    """Single bright pixels on every other row and column, every fifth of them
    among neighbours without an energy; all else exactly at the pedestal."""
    ped = np.full((1, ROWS, COLS), 1000.0, np.float32)
    gain = np.full((1, ROWS, COLS), 25.0, np.float32)
    raw = np.full((1, 1, ROWS, COLS), 1000, np.uint16)
    raw[0, 0, 1:ROWS - 1:2, 1:COLS - 1:2] = 1200
    for k, (r, c) in enumerate((r, c) for r in range(1, ROWS - 1, 2)
                               for c in range(1, COLS - 1, 2)):
        if k % 5 == 0:
            for i, j in NEIGHBOURS[which]:
                gain[0, r + i, c + j] = 1e-39
    ref = oracle.process(oracle.geometry(**GEOM), oracle.thresholds(**THR), ped, gain, raw,
                         want_corrected=True, hit_capacity=ROWS * COLS)
    return ped, gain, raw, ref


@pytest.mark.parametrize("which", list(NEIGHBOURS))
def test_case_reaches_the_compaction(which):
    _, _, raw, ref = _case(which)
    for r0 in range(0, ROWS - 1, BAND):
        assert THREADS < int((raw[0, 0, r0:r0 + BAND] > 1000).sum()) <= LIST
    assert np.isnan(ref.corrected).any()
    assert ref.n_hits == len(ref.hits) == int((raw > 1000).sum())


@pytest.mark.gpu
@pytest.mark.parametrize("which", list(NEIGHBOURS))
def test_seeds_beside_pixels_without_an_energy(which):
    ped, gain, raw, ref = _case(which)
    ctx = pd.pd_create(GEOM, ped, gain, THR)
    assert pd.pd_get_tuning(ctx)["band_rows"] != BAND
    pd.pd_set_tuning(ctx, band_rows=BAND)
    out = pd.process(ctx, pd.frames_to_device(raw), hit_capacity=ROWS * COLS, cm=True)
    torch.cuda.synchronize()
    hits, n = out.hits_host()
    assert n == ref.n_hits
    assert sort_hits(hits).tobytes() == sort_hits(ref.hits).tobytes()
    assert out.cm.cpu().numpy().tobytes() == ref.cm.reshape(1, -1).tobytes()
    np.testing.assert_array_equal(pd.pd_get_summary(ctx)[0], ref.count_map)
