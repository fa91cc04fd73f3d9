"""A scan over a warp needs every lane below a thread in its mask: the mask is
the lanes that exist, not those that __activemask() finds converged after a
branch (the compiler may leave them apart).  Found in the source text."""
from __future__ import annotations

import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1903_06838_gb300", "csrc")


def test_scans_do_not_take_the_active_mask():
    scans = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        with open(path) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"__shfl_up_sync\(\s*(\w+)", text):
            scans += 1
            if m[1].startswith("0x"):
                continue
            # the mask's last definition before the scan
            defs = re.findall(rf"\b{m[1]}\s*=\s*([^;]+);", text[:m.start()])
            assert defs and "activemask" not in defs[-1], (path, m[1], defs[-1:])
    assert scans > 5
