"""A kernel that is launched dependent on the one before may be resident while
that one still writes.  The read-only path (__ldg, ld.global.nc) asks that
memory stays as it is for the kernel's whole life, and the compiler may move
such a load above the wait; so what the kernel before writes is not read that
way.  Found in the source text: no run can show it."""
from __future__ import annotations

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1903_06838_gb300", "csrc")

# file -> names of pointers to what the kernel before writes
WRITTEN = {
    # common-mode values: of a frame, of a module, row and column terms
    "pd_lean.cu": ["cm_frame", "cmf", "cmr", "cmc", "out.cm"],
    "pd_fast.cu": ["cmf", "cmr", "cmc", "out.cm"],
    "pd_matched.cu": ["cmf", "cmr", "cmc", "out.cm"],
    # the weight images, activations and gradient sums of the step's kernels
    "pd_net_train.cu": ["img", "wp", "slices", "dz3", "h2"],
    "pd_net_tc.cu": ["img", "h2"],
}


def test_weight_images_by_explicit_loads():
    # a plain load through a const __restrict__ pointer may become one by the
    # read-only path: the images are read by intrinsics and bulk copies alone
    for name in ("pd_net_train.cu", "pd_net_tc.cu"):
        with open(os.path.join(CSRC, name)) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        assert not re.findall(r"const uint4\*>\(img[^()]*\)\[|\bimg\s*\[(?!i\] =)", text)


@pytest.mark.parametrize("name", list(WRITTEN))
def test_not_through_the_read_only_path(name):
    with open(os.path.join(CSRC, name)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    assert "wait_previous" in text
    loads = re.findall(r"__ldg\(\s*(?:reinterpret_cast<[^>]*>\(\s*)?([\w.]+)", text)
    assert not [v for v in loads if v in WRITTEN[name]]
