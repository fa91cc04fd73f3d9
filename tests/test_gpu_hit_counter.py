"""The hit counter of a call starts at zero whatever it held: cleared by the
common-mode kernel of the bank and row medians, by a memset elsewhere; with the
frames in one chunk, in chunks on one and on two streams, in a recorded graph,
and through the entry that does not allocate.  Reference: the CPU oracle."""
from __future__ import annotations

import pytest

import oracle
from paper_1903_06838_gb300 import pd, synth
from tests._cases import sort_hits

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 5
UNITS = {"banks": dict(n_modules=2, rows=80, cols=128, unit_rows=80, unit_cols=64),
         "rows": dict(n_modules=2, rows=24, cols=128, unit_rows=1, unit_cols=128),
         "odd": dict(n_modules=2, rows=24, cols=45, unit_rows=24, unit_cols=15)}
HOW = {"one_chunk": {}, "one_stream": dict(chunk_frames=2, overlap=0),
       "two_streams": dict(chunk_frames=1, overlap=1), "earlier_pair": dict(kernels=2)}


def _case(units, mode):
    det = synth.Detector(occupancy=0.03, **UNITS[units])
    ped, gain = synth.maps(det)
    raw, _ = synth.frames(det, ped, gain, 0, N, truth=False)
    geom = dict(det.geometry(), cm_mode=mode)
    ref = oracle.process(oracle.geometry(**geom), oracle.thresholds(**det.thresholds()), ped, gain,
                         raw, hit_capacity=raw.size)
    assert ref.n_hits > 0
    ctx = pd.pd_create(geom, ped, gain, det.thresholds())
    dev = pd.frames_to_device(raw)
    return ctx, dev, pd.Outputs(ctx, N, raw.size, cm=True), ref


def _check(out, ref):
    hits, n = out.hits_host()
    assert n == ref.n_hits
    assert sort_hits(hits).tobytes() == sort_hits(ref.hits).tobytes()


@pytest.mark.parametrize("mode", [pd.PD_CM_MEDIAN, pd.PD_CM_NONE, pd.PD_CM_MEAN])
@pytest.mark.parametrize("how", list(HOW))
@pytest.mark.parametrize("units", list(UNITS))
def test_counter_is_cleared(units, how, mode):
    ctx, dev, out, ref = _case(units, mode)
    pd.pd_set_tuning(ctx, **HOW[how])
    for _ in range(3):  # the second and third call find the count of the one before
        pd.pd_process(ctx, dev.data_ptr(), N, 0, **out.ptrs())
    torch.cuda.synchronize()
    _check(out, ref)
    out.n_hits.fill_(0x12345678)
    pd.pd_process(ctx, dev.data_ptr(), N, 0, **out.ptrs())
    torch.cuda.synchronize()
    _check(out, ref)
    out.n_hits.fill_(-1)
    pd.pd_process_noalloc(ctx, dev.data_ptr(), N, 0, **out.ptrs())
    torch.cuda.synchronize()
    _check(out, ref)


@pytest.mark.parametrize("how", ["one_chunk", "two_streams"])
@pytest.mark.parametrize("units", list(UNITS))
def test_counter_is_cleared_in_a_graph(units, how):
    ctx, dev, out, ref = _case(units, pd.PD_CM_MEDIAN)
    pd.pd_set_tuning(ctx, **HOW[how])
    pd.pd_process(ctx, dev.data_ptr(), N, 0, **out.ptrs())
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        pd.pd_process(ctx, dev.data_ptr(), N, 0, **out.ptrs())
    for _ in range(2):
        out.n_hits.fill_(0x12345678)
        graph.replay()
        graph.replay()
        torch.cuda.synchronize()
        _check(out, ref)
