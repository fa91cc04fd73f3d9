"""The band heights that the library's launches choose, from its host code: a
small shared object, compiled on first use beside libpd.so's headers."""
from __future__ import annotations

import atexit
import ctypes
import functools
import os
import shutil
import subprocess
import tempfile

from paper_1903_06838_gb300 import pd

SOURCE = r"""
#include "pd_fast.cuh"
#include "pd_lean.cuh"
static pd::ChainParams params(const uint32_t* g) {
    pd::ChainParams p{};
    p.n_modules = g[0], p.rows = g[1], p.cols = g[2], p.unit_rows = g[3], p.unit_cols = g[4];
    p.cm_mode = g[5], p.hist_bins = g[6];
    p.units_per_row = p.cols / p.unit_cols;
    p.units_per_module = p.rows / p.unit_rows * p.units_per_row;
    p.unit_px = p.unit_rows * p.unit_cols;
    p.module_px = p.rows * p.cols;
    p.frame_px = p.n_modules * p.module_px;
    p.units_per_frame = p.n_modules * p.units_per_module;
    return p;
}
// default height (0: other stencil), height of the call
extern "C" void lean(const uint32_t* g, uint32_t rb, uint32_t frames, int sms, uint32_t* out) {
    const pd::ChainParams p = params(g);
    const pd::LeanConfig lc = pd::make_lean_config(p, rb);
    out[0] = lc.ok ? lc.rb : 0;
    out[1] = lc.ok ? pd::lean_call_rows(p, lc, frames, sms) : 0;
    out[2] = lc.list_cap;
}
extern "C" void band(const uint32_t* g, uint32_t, uint32_t frames, int sms, uint32_t* out) {
    const pd::ChainParams p = params(g);
    const pd::BandConfig bc = pd::make_band_config(p);
    out[0] = bc.ok ? bc.rb : 0;
    out[1] = bc.ok ? pd::band_call_rows(p, bc, frames, sms) : 0;
    out[2] = 0;
}
extern "C" void matched(const uint32_t* g, uint32_t, uint32_t frames, int sms, uint32_t* out) {
    const pd::ChainParams p = params(g);
    out[0] = pd::matched_call_rows(p, 1u << 24, sms);
    out[1] = pd::matched_call_rows(p, frames, sms);
    out[2] = 0;
}
"""


@functools.cache
def _lib():
    lib = pd.build()
    d = tempfile.mkdtemp()
    atexit.register(shutil.rmtree, d, ignore_errors=True)
    src, so = os.path.join(d, "heights.cu"), os.path.join(d, "heights.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.check_call(["nvcc", *pd.ARCH, "-std=c++17", "-O1", "-Xcompiler", "-fPIC", "-shared",
                           "-I", os.path.join(os.path.dirname(lib), "csrc"),
                           "-I", os.path.join(os.path.dirname(os.path.dirname(lib)), "include"),
                           src, "-o", so, lib, "-Xlinker", "-rpath," + os.path.dirname(lib)])
    return ctypes.CDLL(so)


def heights(kind, geometry, frames, sms, band_rows=0, hist_bins=1296):
    """(configured height, height of a call of `frames` frames, entries of the
    candidate list or 0) of the `kind` stencil ("lean", "band", "matched")."""
    g = dict(cm_mode=pd.PD_CM_MEDIAN, **{k: v for k, v in geometry.items() if k != "cm_mode"})
    a = (ctypes.c_uint32 * 7)(*(g[k] for k in ("n_modules", "rows", "cols", "unit_rows",
                                               "unit_cols", "cm_mode")), hist_bins)
    out = (ctypes.c_uint32 * 3)()
    getattr(_lib(), kind)(a, band_rows, frames, sms, out)
    return tuple(out)
