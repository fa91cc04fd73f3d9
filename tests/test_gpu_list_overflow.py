"""Tiles that hold more candidates than the stencils' lists: the lean stencil's
tile and the matched filters' two lists (candidates, and those with a valid
feature) then test every own pixel.  Calls of few tiles take bands too short
for that, so the height is given, or the call is long; each case says how many
a tile of its call holds.  Reference: the CPU oracle, bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1903_06838_gb300 import pd
from tests._cases import sort_hits
from tests._heights import heights

torch = pytest.importorskip("torch")

THR = dict(cm_cut_adu=200.0, zero_thr_kev=0.8, seed_thr_kev=0.8, photon_kev=8.0)
SMS = 152
COLS = 388
LEAN_LIST = 4096                     # candidates of a tile
MATCHED_LIST, MATCHED_VALID = 2048, 1024


def _maps(geom):
    shape = (geom["n_modules"], geom["rows"], geom["cols"])
    return np.full(shape, 1000.0, np.float32), np.full(shape, 25.0, np.float32)


def _bright(frames, geom, row_step, col_step, seed):
    """Single bright pixels on every row_step-th row and col_step-th column
    inside the modules (a few of them of two photons), all else exactly at the
    pedestal."""
    rng = np.random.default_rng(seed)
    raw = np.full((frames, geom["n_modules"], geom["rows"], geom["cols"]), 1000, np.uint16)
    dots = raw[:, :, 1:-1:row_step, 1:-1:col_step]
    dots[...] = rng.choice([1200, 1200, 1200, 1400], dots.shape) + rng.integers(-9, 10, dots.shape)
    return raw


def _reference(geom, raw, bank=None):
    ped, gain = _maps(geom)
    return oracle.process(oracle.geometry(**geom), oracle.thresholds(**THR), ped, gain, raw,
                          hit_capacity=raw.size, want_corrected=True,
                          filters=None if bank is None else oracle.filters(**bank))


def _check(geom, raw, ref, bank=None, band_rows=0):
    ctx = pd.pd_create(geom, *_maps(geom), THR)
    if bank is not None:
        pd.pd_set_filter_bank(ctx, **bank)
    if band_rows:
        pd.pd_set_tuning(ctx, band_rows=band_rows)
        assert pd.pd_get_tuning(ctx)["band_rows"] == band_rows
    out = pd.process(ctx, pd.frames_to_device(raw), hit_capacity=raw.size, corrected=True, cm=True)
    torch.cuda.synchronize()
    hits, n = out.hits_host()
    assert n == ref.n_hits == len(ref.hits)
    assert sort_hits(hits).tobytes() == sort_hits(ref.hits).tobytes()
    assert out.corrected.cpu().numpy().tobytes() == ref.corrected.tobytes()
    for got, exp in zip(pd.pd_get_summary(ctx), (ref.count_map, ref.hist_pix, ref.hist_hit)):
        np.testing.assert_array_equal(got, exp)


# ---- lean stencil ---------------------------------------------------------------
LEAN = dict(n_modules=2, rows=61, cols=COLS, unit_rows=61, unit_cols=COLS // 2)
HEIGHT = 40


def _lean_raw():
    """Random energies and plateaus of equal ones (one seed each), two thirds of
    the first tile's pixels above the threshold."""
    rng = np.random.default_rng(4)
    raw = np.full((2, 2, 61, COLS), 1000, np.uint16)
    raw[:, :, 1:40, :259] = 1000 + rng.integers(60, 180, (2, 2, 39, 259))
    raw[0, :, 5:20, 20:90] = 1150
    raw[1, 1, 41:, 300:] = 1199
    return raw


def test_lean_case_overflows():
    raw = _lean_raw()
    assert heights("lean", LEAN, len(raw), SMS, band_rows=HEIGHT) == (HEIGHT, HEIGHT, LEAN_LIST)
    above = (_reference(LEAN, raw).corrected.reshape(raw.shape) > THR["seed_thr_kev"])
    assert above[:, :, :HEIGHT].sum((2, 3)).min() > LEAN_LIST


@pytest.mark.gpu
def test_lean_tile_tests_every_pixel():
    raw = _lean_raw()
    _check(LEAN, raw, _reference(LEAN, raw), band_rows=HEIGHT)


# ---- matched filters --------------------------------------------------------------
# 640 modules of 48 rows: 1280 tiles of 24 rows, four waves of two an SM
MATCHED = dict(n_modules=16, rows=48, cols=COLS, unit_rows=48, unit_cols=COLS // 2)
FRAMES = 40
TILE = 24


def _bank(binary):
    """One feature, a pixel without signal around it; not binary: its footprint
    weighs 2, so that the valid features are summed and not looked up."""
    f0 = np.zeros((1, 4, 5), np.float32)
    f0[0, 0:3, 1:4] = 1.0
    f0[0, 1, 2] = 0.0
    f1 = np.zeros((1, 4, 5), np.float32)
    f1[0, 1, 2] = 1.0 if binary else 2.0
    return dict(f0=f0, f1=f1, f1_dx=np.zeros_like(f1), f1_dy=np.zeros_like(f1), f1_nmin=[1.0])


#                     rows, columns apart: dots of a tile
MATCHED_CASES = {"valid_list": (2, 3, 12 * 129), "candidate_list": (2, 2, 12 * 193),
                 "both_fit": (2, 6, 12 * 65)}


@pytest.mark.parametrize("case", list(MATCHED_CASES))
def test_matched_case_overflows(case):
    dr, dc, dots = MATCHED_CASES[case]
    assert heights("matched", MATCHED, FRAMES, SMS)[1] == TILE
    raw = _bright(1, MATCHED, dr, dc, 7)
    # a dot is a candidate (signal under F1, none under F0) and valid
    per_tile = [int((raw[0, 0, r:r + TILE] > 1100).sum()) for r in (0, TILE)]
    assert max(per_tile) == dots
    assert (dots > MATCHED_LIST) == (case == "candidate_list")
    assert (dots > MATCHED_VALID) == (case != "both_fit")


@pytest.mark.gpu
@pytest.mark.parametrize("binary", [True, False])
@pytest.mark.parametrize("case", list(MATCHED_CASES))
def test_matched_tile_tests_every_pixel(case, binary):
    dr, dc, _ = MATCHED_CASES[case]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert heights("matched", MATCHED, FRAMES, sms)[1] == TILE
    raw = _bright(FRAMES, MATCHED, dr, dc, 7)
    bank = _bank(binary)
    _check(MATCHED, raw, _reference(MATCHED, raw, bank), bank=bank)
