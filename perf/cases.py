"""The workloads this library is timed on, through its Python binding.

Each case is one call (or one short sequence of calls) that a program using
the library makes over and over: the correction and photon-finding chain on
device-resident frames, the batched launch of a serving slot, the learned
network's inference on a call's hits, and its training step.

Inputs are synthetic, made on the GPU from the seed: pedestal, gain spread,
common-mode offset per unit, noise, and photons whose Gaussian charge cloud
spreads over the 3x3 around the landing pixel (the recipe and the detector
shapes of ``paper_1903_06838_gb300/synth``).

The chain writes its hits in no particular order, so ``run`` puts them in the
order every consumer wants them in, by frame and pixel, with one device sort.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1903_06838_gb300 import filters, pd

PED_MEAN, PED_SIGMA = 1500.0, 40.0       # ADU
ADU_PER_KEV, GAIN_SIGMA = 25.0, 0.03
NOISE_SIGMA, CM_SIGMA = 4.0, 15.0        # ADU
CLOUD_SIGMA = 0.3                        # pixel pitches
THRESHOLD_KEV = 5.0 * NOISE_SIGMA / ADU_PER_KEV  # of signal and of seeds: 5 sigma
GAIN_SHIFT = 14                          # auto-ranging words: stage in the top two bits
STAGE_GAIN = (1.0, 1.0 / 3.0, 1.0 / 100.0)
STAGE_PED = (0.0, -300.0, -700.0)
BLOBS, BLOB_KEV = 3, 3000.0              # bright spots per module (auto-ranging)

CM_MODE = {"median": pd.PD_CM_MEDIAN, "none": pd.PD_CM_NONE, "mean": pd.PD_CM_MEAN,
           "stacked": pd.PD_CM_MEAN_STACKED}

# the detector shapes of the generator's presets
EPIX = dict(modules=1, rows=704, cols=768, unit_rows=1, unit_cols=384, kev=6.0)
ASIC = dict(modules=1, rows=352, cols=384, unit_rows=1, unit_cols=384, kev=8.0)
ASIC16 = dict(modules=16, rows=352, cols=384, unit_rows=1, unit_cols=384, kev=12.0)
CSPAD = dict(modules=32, rows=185, cols=388, unit_rows=185, unit_cols=194, kev=8.0)

NET_BATCH = 65536   # patches per chunk of the network's buffers
NO_HIT = -(1 << 30)  # pixel of an unused hit record
TRAIN_SET = 65536   # hits of the training set a step draws its rows from


def _chain(shape, frames, occ_lo, occ_hi, **kw):
    return dict(kind="chain", **shape, frames=frames, occ_lo=occ_lo, occ_hi=occ_hi,
                **{**dict(cm="median", paper_order=False, matched=False, stages=0,
                          hits=True, corrected=False, summary=False, graph=False), **kw})


def listed():
    return [
        # one frame of a live view (the corrected frame, the photon count but no
        # hit list): the smallest call, bound by launches
        dict(_chain(EPIX, 1, 0.01, 0.01, hits=False, corrected=True), name="epix_frame"),
        # a burst of one ASIC at low flux, a latency-bound loop's pass (recorded
        # once as a graph, as such a loop is)
        dict(_chain(ASIC, 16, 0.0015, 0.0015, graph=True), name="asic_burst"),
        # what one slot of the streaming server holds: 80 % / 20 % of two
        # detectors, in one captured batch
        dict(kind="slot", epix_frames=15, cspad_frames=4, occ_lo=0.001, occ_hi=0.02,
             name="serve_slot"),
        # the benchmark's chain: a batch of the 2.2 Mpixel detector
        dict(_chain(CSPAD, 256, 0.005, 0.005), name="cspad_batch"),
        # the same detector with the corrected frames kept (calibration, inspection)
        dict(_chain(CSPAD, 21, 0.005, 0.005, corrected=True), name="cspad_corrected"),
        # sixteen ASICs at varying, partly high flux: a third of the mixed batch
        dict(_chain(ASIC16, 45, 0.001, 0.1), name="asic16_bright"),
        # the paper's three stacked common-mode stages
        dict(_chain(CSPAD, 64, 0.005, 0.005, cm="stacked"), name="cspad_stacked"),
        # the paper's matched filters in place of the 3x3 local maximum
        dict(_chain(CSPAD, 64, 0.005, 0.005, matched=True), name="cspad_matched"),
        # an auto-ranging detector: three gain stages in the raw words
        dict(_chain(CSPAD, 64, 0.005, 0.005, stages=3), name="cspad_autorange"),
        # a small sensor with odd sizes in the paper's order (gain first, mean
        # common mode), with the run's summaries read at its end
        dict(_chain(dict(modules=4, rows=185, cols=291, unit_rows=185, unit_cols=97, kev=8.0),
                    51, 0.005, 0.02, cm="mean", paper_order=True, summary=True),
             name="paper_order_run"),
        # the learned refinement's inference on the hits of a burst
        dict(kind="infer", **EPIX, frames=48, occ_lo=0.005, occ_hi=0.05, name="net_infer"),
        # one training step's rows and gradients at the trainer's batch size
        dict(kind="train", hits=2048, name="net_train"),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(_log_uniform(rng, lo, hi)))))


def draw(rng):
    """A random case of the listed ones' ranges."""
    kind = rng.choices(["chain", "odd", "slot", "infer", "train"], [8, 4, 2, 3, 3])[0]
    occ_lo = round(_log_uniform(rng, 0.001, 0.02), 5)
    occ_hi = rng.choice([occ_lo, round(min(0.1, occ_lo * rng.uniform(2.0, 10.0)), 5)])
    if kind == "slot":
        return dict(kind="slot", epix_frames=_log_int(rng, 1, 32),
                    cspad_frames=_log_int(rng, 1, 16), occ_lo=occ_lo, occ_hi=occ_hi)
    if kind == "infer":
        shape = rng.choice([EPIX, ASIC])
        return dict(kind="infer", **shape, frames=_log_int(rng, 1, 60), occ_lo=occ_lo,
                    occ_hi=occ_hi)
    if kind == "train":
        return dict(kind="train", hits=_log_int(rng, 100, 8192))
    mode = rng.choices(["plain", "none", "mean", "stacked", "matched", "autorange", "paper"],
                       [6, 1, 2, 2, 2, 2, 1])[0]
    kw = dict(plain={}, none=dict(cm="none"), mean=dict(cm="mean"), stacked=dict(cm="stacked"),
              matched=dict(matched=True), autorange=dict(stages=rng.choice([2, 3])),
              paper=dict(cm=rng.choice(["median", "mean", "stacked"]), paper_order=True))[mode]
    if rng.random() < 0.2:
        kw = dict(kw, corrected=True, hits=rng.random() < 0.5)
    if kind == "odd":
        # any size of sensor: whole-height banks, blocks or rows as units
        units_x = rng.choice([1, 1, 2, 3])
        rows, ucols = rng.randint(24, 400), rng.randint(24, 520 // units_x)
        shape = dict(modules=rng.randint(1, 6), rows=rows, cols=ucols * units_x,
                     unit_rows=rng.choice([rows, rows, 1]), unit_cols=ucols,
                     kev=rng.choice([6.0, 8.0, 12.0]))
    else:
        shape = rng.choice([EPIX, ASIC, ASIC16, CSPAD, CSPAD])
    px = shape["modules"] * shape["rows"] * shape["cols"]
    most = 8_000_000 if mode == "paper" else 24_000_000 if kind == "odd" else \
        300_000_000 if mode in ("plain", "none") else 90_000_000
    if "corrected" in kw:
        most = min(most, 60_000_000)
    if occ_hi > 0.02:
        most = min(most, 80_000_000)
    return _chain(shape, _log_int(rng, 1, max(1, min(256, most // px))), occ_lo, occ_hi, **kw)


# ---- inputs -------------------------------------------------------------------
def _pixels(case):
    return case["modules"] * case["rows"] * case["cols"]


def _units(case):
    return case["modules"] * (case["rows"] // case["unit_rows"]) * \
        (case["cols"] // case["unit_cols"])


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _maps(case, g):
    """Pedestal (ADU) and gain (ADU/keV), float32 [modules, rows, cols]."""
    shape = (case["modules"], case["rows"], case["cols"])
    ped = PED_MEAN + PED_SIGMA * torch.randn(shape, generator=g, device="cuda")
    gain = ADU_PER_KEV * (1.0 + GAIN_SIGMA * torch.randn(shape, generator=g, device="cuda"))
    return ped, gain


def _photons(case):
    """Photons of each frame: occupancies spread evenly over the logarithm of
    the case's range, so that their total is the case's own."""
    n, px = case["frames"], _pixels(case)
    lo, hi = math.log(case["occ_lo"]), math.log(case["occ_hi"])
    return [int(px * math.exp(lo + (hi - lo) * (i + 0.5) / n)) for i in range(n)]


def _capacity(case):
    """Hit records of the call's buffer."""
    if not case.get("hits", True):
        return 0
    photons = sum(_photons(case))
    cap = photons + photons // 50 + 64
    if case.get("matched"):
        cap += cap // 4
    if case.get("stages"):
        cap += 250 * case["frames"] * case["modules"]
    return cap


def _charge(case, counts, g):
    """Photon energy deposited in each pixel, keV [n, modules, rows, cols]."""
    n, M, R, C = counts.numel(), case["modules"], case["rows"], case["cols"]
    px, total = M * R * C, int(counts.sum())
    frame = torch.repeat_interleave(torch.arange(n, device="cuda"), counts)
    at = torch.randint(0, px, (total,), generator=g, device="cuda")
    uv = torch.rand((2, total), generator=g, device="cuda")
    axis = []
    for k in range(2):  # share of the cloud in the three pixels of each axis
        edge = torch.arange(-1.0, 3.0, device="cuda")[:, None] - uv[k][None]
        cdf = torch.special.erf(edge / (CLOUD_SIGMA * math.sqrt(2.0)))
        share = cdf[1:] - cdf[:-1]
        axis.append(share / share.sum(0))
    row, col = (at // C) % R, at % C
    # summed in 64 bits: the order of the additions then never shows in the words
    out = torch.zeros(n * px, device="cuda", dtype=torch.float64)
    base = frame * px + at
    for i in (-1, 0, 1):
        for j in (-1, 0, 1):
            ok = (row + i >= 0) & (row + i < R) & (col + j >= 0) & (col + j < C)
            kev = case["kev"] * axis[0][i + 1] * axis[1][j + 1]
            out.index_add_(0, (base + i * C + j)[ok], kev[ok].double())
    return out.float().view(n, M, R, C)


def _frames(case, n, ped, gain, g):
    """Raw frames (int16 holding the uint16 bits)."""
    M, R, C = case["modules"], case["rows"], case["cols"]
    ur, uc = case["unit_rows"], case["unit_cols"]
    counts = torch.tensor(_photons(case), device="cuda")
    counts = counts[torch.randperm(n, generator=g, device="cuda")]
    raw = torch.empty((n, M, R, C), dtype=torch.int16, device="cuda")
    step = max(1, 16_000_000 // (M * R * C))
    for a in range(0, n, step):
        b = min(n, a + step)
        charge = _charge(case, counts[a:b], g)
        if case.get("stages"):
            charge += _bright_spots(case, b - a, g)
        off = CM_SIGMA * torch.randn((b - a, M, R // ur, 1, C // uc, 1), generator=g,
                                     device="cuda")
        off = off.expand(-1, -1, -1, ur, -1, uc).reshape(b - a, M, R, C)
        noise = NOISE_SIGMA * torch.randn((b - a, M, R, C), generator=g, device="cuda")
        v = ped + charge * gain + off + noise
        if case.get("stages"):
            w = _ranged(case, v, charge, ped, gain, g)
        else:
            w = v.round().clamp(0, 65535).to(torch.int32)
        raw[a:b] = w.to(torch.int16)
    return raw


def _bright_spots(case, n, g):
    """Bright Gaussian spots on every module, keV per pixel."""
    M, R, C = case["modules"], case["rows"], case["cols"]
    y = torch.arange(R, device="cuda").view(R, 1)
    x = torch.arange(C, device="cuda").view(1, C)
    out = torch.zeros((n, M, R, C), device="cuda")
    for _ in range(BLOBS):
        u = torch.rand((4, n, M, 1, 1), generator=g, device="cuda")
        cy, cx, w = u[0] * R, u[1] * C, 1.5 + 4.5 * u[2]
        ry, rx = (y - cy) ** 2 / (2 * w * w), (x - cx) ** 2 / (2 * w * w)
        out += (0.05 + 0.95 * u[3]) * BLOB_KEV * torch.exp(-ry) * torch.exp(-rx)
    return out


def _ranged(case, v, charge, ped, gain, g):
    """Auto-ranging words: a pixel past 90 % of the ADC range takes the next
    stage; a few words carry an invalid stage."""
    full = (1 << GAIN_SHIFT) - 1
    stage = torch.zeros(v.shape, dtype=torch.int32, device="cuda")
    for k in range(1, case["stages"]):
        up = v > 0.9 * full
        lower = ped + STAGE_PED[k] + charge * gain * STAGE_GAIN[k] + \
            NOISE_SIGMA * torch.randn(v.shape, generator=g, device="cuda")
        stage = torch.where(up, k, stage)
        v = torch.where(up, lower, v)
    w = (stage << GAIN_SHIFT) | v.round().clamp(0, full).to(torch.int32)
    bad = torch.rand(v.shape, generator=g, device="cuda") < 1e-4
    return torch.where(bad & (case["stages"] < 4), (case["stages"] << GAIN_SHIFT) | (w & full), w)


def _thresholds(case):
    return dict(cm_cut_adu=case["kev"] * ADU_PER_KEV, zero_thr_kev=THRESHOLD_KEV,
                seed_thr_kev=THRESHOLD_KEV, photon_kev=case["kev"])


def _context(case, ped, gain):
    geometry = dict(n_modules=case["modules"], rows=case["rows"], cols=case["cols"],
                    unit_rows=case["unit_rows"], unit_cols=case["unit_cols"],
                    cm_mode=CM_MODE[case.get("cm", "median")],
                    cm_after_gain=int(case.get("paper_order", False)))
    stages = case.get("stages", 0)
    if stages:
        ped = torch.stack([ped + STAGE_PED[k] for k in range(stages)])
        gain = torch.stack([gain * STAGE_GAIN[k] for k in range(stages)])
    ctx = pd.pd_create(geometry, ped.cpu().numpy(), gain.cpu().numpy(), _thresholds(case),
                       n_gains=stages, gain_shift=GAIN_SHIFT if stages else 0)
    if case.get("matched"):
        pd.pd_set_filter_bank(ctx, **filters.example_bank())
    return ctx


def _outputs(case, ctx, n):
    """Device buffers of one call; unused hit records hold pixel NO_HIT and
    zeros, so that they sort in front."""
    out = pd.Outputs(ctx, n, _capacity(case), corrected=case.get("corrected", False), cm=True)
    rec = out.hits.view(torch.int32)
    rec.zero_()
    rec[:, 1] = NO_HIT
    return out


def _ordered(hits, keys):
    """Hit records in the order of their keys, int32 [records, 6]."""
    order = torch.sort(keys).indices
    return torch.index_select(hits.view(torch.int64), 0, order).view(torch.int32)


def _hits(rec):
    return dict(where=rec[:, :2], energy_dx_dy=rec.view(torch.float32)[:, 2:5],
                count_npix_flags=rec[:, 5])


class _Part:
    """One detector's frames, context and output buffers."""

    def __init__(self, case, seed):
        g = _generator(seed)
        self.n = case["frames"]
        self.ped, self.gain = _maps(case, g)
        self.raw = _frames(case, self.n, self.ped, self.gain, g)
        self.ctx = _context(case, self.ped, self.gain)
        self.px = _pixels(case)
        self.out = _outputs(case, self.ctx, self.n)

    def process(self):
        pd.pd_process(self.ctx, self.raw.data_ptr(), self.n, 0, **self.out.ptrs())

    def keys(self):
        """Place of every hit record in the order of frames and pixels."""
        rec = self.out.hits.view(torch.int32)
        return torch.add(rec[:, 1], rec[:, 0], alpha=self.px)

    def results(self):
        out = dict(n_hits=self.out.n_hits, cm=self.out.cm)
        if self.out.hit_capacity:
            out.update(_hits(_ordered(self.out.hits, self.keys())))
        if self.out.corrected is not None:
            out["corrected"] = self.out.corrected
        return out


def _slot_parts(case):
    occ = dict(occ_lo=case["occ_lo"], occ_hi=case["occ_hi"])
    return dict(EPIX, frames=case["epix_frames"], **occ), \
        dict(CSPAD, frames=case["cspad_frames"], **occ)


def _infer_hits(case):
    return max(1, int(0.6 * sum(_photons(case))))


def _prepare_infer(case, seed):
    part = _Part(case, seed)
    part.process()
    # as many hits as every seed gives (photons that share a 3x3 merge)
    n = _infer_hits(case)
    assert int(part.out.n_hits.item()) >= n
    hits = _ordered(part.out.hits, part.keys())[-n:].contiguous()
    net = pd.pd_net_create(NET_BATCH, seed & 0xFFFF)
    return dict(kind="infer", part=part, n=n, hits=hits, net=net,
                patches=torch.empty((n, 25), device="cuda"), out=torch.empty((n, 7), device="cuda"))


def _training_set(n, g):
    """Patches of one to four photons around the seed pixel (in photon
    energies, noise included), their counts, offsets and offset mask."""
    count = 1 + torch.poisson(torch.full((n,), 0.3, device="cuda"), generator=g).clamp(max=3)
    x = torch.zeros((n, 5, 5), device="cuda")
    first = None
    for k in range(4):
        u = torch.rand((2, n), generator=g, device="cuda")
        if k == 0:
            first = u - 0.5
        axis = []
        for i in range(2):
            edge = torch.arange(6.0, device="cuda")[None] - 2.0 - u[i][:, None]
            cdf = torch.special.erf(edge / (CLOUD_SIGMA * math.sqrt(2.0)))
            axis.append(0.5 * (cdf[:, 1:] - cdf[:, :-1]))
        x += (count > k).view(n, 1, 1) * axis[1][:, :, None] * axis[0][:, None, :]
    sigma = NOISE_SIGMA / ADU_PER_KEV / 8.0
    x += sigma * torch.randn(x.shape, generator=g, device="cuda")
    mask = (count == 1).to(torch.uint8)
    targets = (first * mask).t().contiguous()
    return x.reshape(n, 25), count.to(torch.uint8), targets, mask


def _prepare_train(case, seed):
    g, n = _generator(seed), case["hits"]
    full = _training_set(TRAIN_SET, g)
    idx = torch.randint(0, TRAIN_SET, (n,), generator=g, device="cuda", dtype=torch.int32)
    rows = (torch.empty((n, 25), device="cuda"), torch.empty(n, dtype=torch.uint8, device="cuda"),
            torch.empty((n, 2), device="cuda"), torch.empty(n, dtype=torch.uint8, device="cuda"))
    return dict(kind="train", n=n, full=full, idx=idx, rows=rows,
                n_reg=float(full[3][idx.long()].sum()), net=pd.pd_net_create(8192, seed & 0xFFFF),
                grads=torch.empty(pd.pd_net_num_params(), device="cuda"),
                loss=torch.zeros(1, device="cuda"))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "infer":
        return _prepare_infer(case, seed)
    if kind == "train":
        return _prepare_train(case, seed)
    if kind == "slot":
        parts = [_Part(c, seed + k) for k, c in enumerate(_slot_parts(case))]
        # the slot's hits in one buffer, the second detector's after the first's
        hits = torch.cat([q.out.hits for q in parts])
        cut = len(parts[0].out.hits)
        parts[0].out.hits, parts[1].out.hits = hits[:cut], hits[cut:]
        batch = pd.pd_batch_create(len(parts))
        items = [(q.ctx, q.raw.data_ptr(), q.n, 0, q.out) for q in parts]
        stream = torch.cuda.Stream()
        pd.pd_batch_capture(batch, items, stream)
        return dict(kind="slot", parts=parts, batch=batch, hits=hits)
    state = dict(kind="chain", part=_Part(case, seed), summary=case["summary"], graph=None)
    if case["graph"]:
        _record(state)
    return state


def _record(state):
    """The pass of a latency-bound loop as a CUDA graph."""
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        run(state)
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = run(state)
    state.update(graph=graph, out=out)


# ---- one pass -----------------------------------------------------------------
def run(state):
    kind = state["kind"]
    if kind == "chain":
        part = state["part"]
        if state["graph"]:
            state["graph"].replay()
            return state["out"]
        if state["summary"]:
            pd.pd_reset_summary(part.ctx)
        part.process()
        out = part.results()
        if state["summary"]:
            count_map, hist_pix, hist_hit = pd.pd_get_summary(part.ctx)
            out.update(count_map=count_map.view(np.int32), hist_pix=hist_pix.view(np.int64),
                       hist_hit=hist_hit.view(np.int64))
        return out
    if kind == "slot":
        pd.pd_batch_replay(state["batch"])
        a, b = state["parts"]
        keys = torch.cat([a.keys(), b.keys() + a.n * a.px])
        return dict(_hits(_ordered(state["hits"], keys)), n_hits=[a.out.n_hits, b.out.n_hits],
                    cm=[a.out.cm, b.out.cm])
    if kind == "infer":
        part, n = state["part"], state["n"]
        pd.pd_net_gather(part.ctx, part.raw.data_ptr(), 0, part.out.cm.data_ptr(),
                         state["hits"].data_ptr(), n, state["patches"].data_ptr())
        pd.pd_net_forward(state["net"], state["patches"].data_ptr(), n, state["out"].data_ptr())
        return dict(patches=state["patches"], out=state["out"])
    rows, n = state["rows"], state["n"]
    state["loss"].zero_()
    pd.pd_net_take(*(t.data_ptr() for t in state["full"]), state["idx"].data_ptr(), n,
                   *(t.data_ptr() for t in rows))
    pd.pd_net_gradients(state["net"], *(t.data_ptr() for t in rows), n, state["n_reg"], 10.0,
                        state["grads"].data_ptr(), state["loss"].data_ptr())
    return dict(grads=state["grads"], loss=state["loss"])


# ---- what a pass cannot do without ----------------------------------------------
def _chain_bytes(case):
    px, n = _pixels(case), case["frames"]
    hits = sum(_photons(case)) if case.get("hits", True) else 0
    maps = 8.0 * px * max(1, case.get("stages", 0))
    cm = 4.0 * n * _units(case)
    if case.get("cm") == "stacked":
        cm += 4.0 * n * case["modules"] * (case["rows"] + case["cols"])
    return 2.0 * px * n + maps + 24.0 * hits + cm + \
        (4.0 * px * n if case.get("corrected") else 0.0) + (4.0 * px if case.get("summary") else 0.0)


# multiply-adds of the network's forward pass per hit, times two
NET_FLOPS = 2.0 * (25 * 32 * 9 + 25 * 32 * 288 + 64 * 800 + 7 * 64)


def work(case):
    kind = case["kind"]
    if kind == "slot":
        parts = _slot_parts(case)
        return {"bytes": sum(_chain_bytes(c) for c in parts),
                "flops": sum(12.0 * _pixels(c) * c["frames"] for c in parts)}
    if kind == "infer":
        n = _infer_hits(case)
        # a hit record, the raw words and maps of its 5x5, the patch and the outputs
        return {"bytes": n * (24.0 + 25 * 10.0 + 100.0 + 28.0), "flops": n * NET_FLOPS}
    if kind == "train":
        n = case["hits"]
        return {"bytes": n * (100.0 + 8.0 + 2.0 + 4.0) + 2 * 4.0 * 61287, "flops": 3.0 * n * NET_FLOPS}
    # dark, common mode, gain, threshold, histogram bin and comparison per pixel
    return {"bytes": _chain_bytes(case), "flops": 12.0 * _pixels(case) * case["frames"]}


# ---- the same in 64 bits --------------------------------------------------------
def _shift(s, i, j):
    """s at (row + i, col + j), zero outside the module."""
    R, C = s.shape[-2:]
    out = torch.zeros_like(s)
    if abs(i) < R and abs(j) < C:
        out[..., max(0, -i):R - max(0, i), max(0, -j):C - max(0, j)] = \
            s[..., max(0, i):R + min(0, i), max(0, j):C + min(0, j)]
    return out


def _mean_of(v, cut, dims, group):
    sel = v < cut
    total = torch.where(sel, v, 0.0).sum(dims, keepdim=True)
    return total / sel.sum(dims, keepdim=True).double().clamp(min=math.sqrt(group))


def _median_of(v, cut, group):
    """Lower median of v below the cut over the last dimension; NaN stays out."""
    need = math.ceil(math.sqrt(group))
    srt = torch.where(v < cut, v, math.inf).sort(-1).values
    cnt = torch.isfinite(srt).sum(-1, keepdim=True)
    med = srt.gather(-1, ((cnt - 1) // 2).clamp(min=0))
    return torch.where(cnt >= max(need, 1), med, 0.0)


def _exact_energy(case, raw, ped, gain):
    """(common mode [n, values], e [n, modules, rows, cols]) of some frames."""
    n, M, R, C = raw.shape
    ur, uc = case["unit_rows"], case["unit_cols"]
    w = raw.to(torch.int64) & 0xFFFF
    ig = 1.0 / gain.double()
    ordered = case.get("paper_order", False)
    cut = case["kev"] if ordered else case["kev"] * ADU_PER_KEV
    stages = case.get("stages", 0)
    if stages:
        stage, val = w >> GAIN_SHIFT, (w & ((1 << GAIN_SHIFT) - 1)).double()
        d = val - ped.double()
        selected = torch.where(stage == 0, d, math.nan)
    else:
        d = w.double() - ped.double()
        if ordered:
            d = d * ig
        selected = d
    mode = case.get("cm", "median")
    blocks = (n, M, R // ur, ur, C // uc, uc)
    cms = []
    if mode == "none":
        cms.append(torch.zeros((n, _units(case)), device=raw.device, dtype=torch.float64))
        c = d
    else:
        if mode == "median":
            flat = selected.view(blocks).permute(0, 1, 2, 4, 3, 5).reshape(n, -1, ur * uc)
            cm = _median_of(flat, cut, ur * uc).view(n, M, R // ur, 1, C // uc, 1)
        else:
            cm = _mean_of(selected.view(blocks), cut, (3, 5), ur * uc)
        cms.append(cm.reshape(n, -1))
        c = (d.view(blocks) - cm).view(n, M, R, C)
        if mode == "stacked":
            for dim, size in ((3, C), (2, R)):
                cm = _mean_of(c, cut, (dim,), size)
                cms.append(cm.reshape(n, -1))
                c = c - cm
    e = c if ordered else c * ig
    if stages:
        e = torch.where(stage == 0, e, 0.0)
        for k in range(1, stages):
            # the maps as the program hands them over, in 32 bits
            pk, gk = (ped + STAGE_PED[k]).double(), (gain * STAGE_GAIN[k]).double()
            e = torch.where(stage == k, (val - pk) / gk, e)
    return torch.cat(cms, 1), e


def _exact_hits(case, e):
    """energy, dx, dy of the hits of some frames in order, [hits, 3]."""
    s = torch.where(e > THRESHOLD_KEV, e, 0.0)
    E, mx, my = torch.zeros_like(s), torch.zeros_like(s), torch.zeros_like(s)
    if case.get("matched"):
        bank = filters.example_bank()
        on = (s > 0).double()
        seed = torch.zeros(s.shape, dtype=torch.bool, device=s.device)

        def taps(a, f):
            got = torch.zeros_like(s)
            for i in range(4):
                for j in range(5):
                    if f[i, j]:
                        got += float(f[i, j]) * _shift(a, i - 1, j - 2)
            return got
        for f0, f1, fx, fy, nmin in zip(*(bank[k] for k in ("f0", "f1", "f1_dx", "f1_dy",
                                                            "f1_nmin"))):
            drop = taps(s, f1)
            valid = (taps(on, f0) == 0) & (taps(on, f1) >= float(nmin))
            use = valid & (drop != 0)
            E += torch.where(valid, drop, 0.0)
            mx += torch.where(use, taps(s, fx) / drop, 0.0)
            my += torch.where(use, taps(s, fy) / drop, 0.0)
            seed |= valid
        seed &= E != 0
    else:
        seed = s > THRESHOLD_KEV
        for i in (-1, 0, 1):
            for j in (-1, 0, 1):
                q = _shift(s, i, j)
                if (i, j) < (0, 0):
                    seed &= s > q
                elif (i, j) > (0, 0):
                    seed &= s >= q
                E += q
                mx += j * q
                my += i * q
        mx, my = mx / E, my / E
    hit = seed & (torch.round(E / case["kev"]) >= 1)
    return torch.stack([E[hit], mx[hit], my[hit]], 1)


def _exact_part(case, seed):
    g = _generator(seed)
    ped, gain = _maps(case, g)
    raw = _frames(case, case["frames"], ped, gain, g)
    step = max(1, 24_000_000 // _pixels(case))
    cms, hits, es = [], [], []
    for a in range(0, case["frames"], step):
        cm, e = _exact_energy(case, raw[a:a + step], ped, gain)
        cms.append(cm)
        if case.get("hits", True):
            hits.append(_exact_hits(case, e))
        if case.get("corrected"):
            es.append(e.reshape(e.shape[0], -1))
    out = dict(n_hits=None, cm=torch.cat(cms))
    if hits:
        hits = torch.cat(hits)
        full = torch.zeros((_capacity(case), 3), dtype=torch.float64, device="cuda")
        full[len(full) - len(hits):] = hits
        # frames, pixels, counts and flags are whole numbers: no value here
        out.update(where=None, energy_dx_dy=full, count_npix_flags=None)
    if es:
        out["corrected"] = torch.cat(es)
    if case.get("summary"):
        out.update(count_map=None, hist_pix=None, hist_hit=None)
    return out


def _net_parameters(net):
    w = torch.from_numpy(pd.pd_net_get_params(net)).cuda().double()
    sizes = [(32, 9), (32,), (32, 9, 32), (32,), (64, 25 * 32), (64,), (7, 64), (7,)]
    out, at = [], 0
    for s in sizes:
        k = math.prod(s)
        out.append(w[at:at + k].view(s).clone().requires_grad_())
        at += k
    return out


def _net_forward(params, x):
    w1, b1, w2, b2, w3, b3, w4, b4 = params
    n = x.shape[0]

    def columns(a):  # [n, 25, channels] -> [n, 25, 9, channels]
        grid = torch.nn.functional.pad(a.view(n, 5, 5, -1), (0, 0, 1, 1, 1, 1))
        return torch.stack([grid[:, i:i + 5, j:j + 5].reshape(n, 25, -1)
                            for i in range(3) for j in range(3)], 2)
    h = torch.relu(columns(x.view(n, 25, 1)).squeeze(-1) @ w1.t() + b1)
    h = torch.relu(columns(h).reshape(n, 25, 288) @ w2.reshape(32, 288).t() + b2)
    h = torch.relu(h.reshape(n, 800) @ w3.t() + b3)
    return h @ w4.t() + b4


def exact(case, seed):
    kind = case["kind"]
    if kind == "chain":
        return _exact_part(case, seed)
    if kind == "slot":
        a, b = (_exact_part(c, seed + k) for k, c in enumerate(_slot_parts(case)))
        # unused records of both detectors come first
        rows = [q["energy_dx_dy"][q["energy_dx_dy"][:, 0] != 0] for q in (a, b)]
        full = torch.zeros((len(a["energy_dx_dy"]) + len(b["energy_dx_dy"]), 3),
                           dtype=torch.float64, device="cuda")
        full[len(full) - len(rows[0]) - len(rows[1]):] = torch.cat(rows)
        return dict(where=None, energy_dx_dy=full, count_npix_flags=None, n_hits=[None, None],
                    cm=[a["cm"], b["cm"]])
    state = prepare(case, seed)
    params = _net_parameters(state["net"])
    if kind == "infer":
        # the 5x5 of e / photon energy around each hit's seed
        part, px = state["part"], _pixels(case)
        R, C = case["rows"], case["cols"]
        hits = state["hits"].long()
        got = []
        step = max(1, 24_000_000 // px)
        for a in range(0, part.n, step):
            _, e = _exact_energy(case, part.raw[a:a + step], part.ped, part.gain)
            h = hits[(hits[:, 0] >= a) & (hits[:, 0] < a + step)]
            grid = torch.nn.functional.pad(e / case["kev"], (2, 2, 2, 2))
            m, r, c = h[:, 1] // (R * C), h[:, 1] // C % R, h[:, 1] % C
            got.append(torch.stack([grid[h[:, 0] - a, m, r + i, c + j]
                                    for i in range(5) for j in range(5)], 1))
        patches = torch.cat(got)
        with torch.no_grad():
            out = torch.cat([_net_forward(params, q) for q in patches.split(8192)])
        return dict(patches=patches, out=out)
    rows = [t[state["idx"].long()] for t in state["full"]]
    out = _net_forward(params, rows[0].double())
    keep = rows[3].double().view(-1, 1)
    loss = torch.nn.functional.cross_entropy(out[:, :5], rows[1].long().clamp(max=4)) + \
        10.0 * (((out[:, 5:] - rows[2].double()) * keep) ** 2).sum() / max(1.0, state["n_reg"])
    grads = torch.autograd.grad(loss, params)
    return dict(grads=torch.cat([q.reshape(-1) for q in grads]), loss=loss.detach().view(1))
