"""The band height of a call: the default for calls of many tiles, less for
calls of few, never more, and an explicit height as it was given."""
from __future__ import annotations

import math

import pytest

from tests._heights import heights

SMS = 152
SHAPES = {
    "lean": [dict(n_modules=1, rows=704, cols=768, unit_rows=1, unit_cols=384),
             dict(n_modules=32, rows=185, cols=388, unit_rows=185, unit_cols=194),
             dict(n_modules=2, rows=97, cols=64, unit_rows=1, unit_cols=64)],
    "band": [dict(n_modules=4, rows=185, cols=291, unit_rows=185, unit_cols=97),
             dict(n_modules=1, rows=352, cols=384, unit_rows=1, unit_cols=384)],
    "matched": [dict(n_modules=32, rows=185, cols=388, unit_rows=185, unit_cols=194),
                dict(n_modules=1, rows=352, cols=384, unit_rows=1, unit_cols=384)],
}
CASES = [(k, g) for k, gs in SHAPES.items() for g in gs]
IDS = [f"{k}_{g['rows']}x{g['cols']}" for k, g in CASES]


@pytest.mark.parametrize("kind,geometry", CASES, ids=IDS)
def test_height_of_a_call(kind, geometry):
    rows = geometry["rows"]
    default = heights(kind, geometry, 1, SMS)[0]
    assert 1 < default <= rows
    got = [heights(kind, geometry, n, SMS)[1] for n in (1, 2, 3, 5, 9, 20, 50, 120, 10 ** 5)]
    assert all(1 <= h <= default for h in got)
    assert got[-1] == default
    if geometry["n_modules"] * math.ceil(rows / default) < SMS:  # not one tile an SM
        assert got[0] < default


@pytest.mark.parametrize("geometry", SHAPES["lean"], ids=[i for i in IDS if i[:4] == "lean"])
def test_explicit_height_is_kept(geometry):
    default = heights("lean", geometry, 1, SMS)[0]
    for height in (1, 5, default - 1, default + 1):
        if height > geometry["rows"]:
            continue
        for frames in (1, 40, 10 ** 5):
            assert heights("lean", geometry, frames, SMS, band_rows=height)[:2] == (height, height)
