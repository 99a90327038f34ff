"""Benchmark: DeGraF detection + RLOF tracking on a 1242x375 driving-scene-shaped pair.

One step = one pass of the whole hot path over one frame pair: DeGraF detection
on frame 1 (window 7, step 3: 50,676 points), the 5-level pyramids of both frames,
and RLOF tracking of every point (11x11 support, max 30 iterations, gain/offset
model, FP32). Frames are seeded synthetic uint8 pairs (radial expansion up to
150 px plus three moving rectangles) standing in for KITTI.

Prints one JSON line. `value` is tracked points per second over the whole job
(device-resident inputs, CUDA events, L2 flushed between steps); `e2e` is the
same metric through the public host-buffer API with the copies in the timed
region. `--impl reference` times the FP64 CPU oracle instead.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import subprocess
import sys
import tempfile
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import synth  # noqa: E402

METRIC = "tracked points/s and frame pairs/s at 1242x375; % HBM roofline; EPE vs FP64 oracle"
WORKLOAD = dict(workload="driving-scene pair 1242x375: DeGraF w=7 step=3 (50676 pts) + RLOF "
                "5 levels 11x11 max 30 iters gain/offset model, FP32",
                W=1242, H=375, win=7, step=3, levels=5, radius=5, max_iter=30, model=4)
L2_FLUSH_BYTES = 256 << 20


def _measured_peaks():
    """HBM bandwidth and maximum SM clock measured on the GB300s
    (MEASURED_PEAKS.json), else the stated fallback (6.8 TB/s, 2070 MHz)."""
    try:
        rec = json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
        return float(rec["hbm_gbs"]), float(rec.get("sm_max_mhz", 2070.0)), "measured (MEASURED_PEAKS.json)"
    except (OSError, ValueError, KeyError, TypeError):
        return 6800.0, 2070.0, "fallback (no MEASURED_PEAKS.json)"


HBM_PEAK_GBS, SM_MAX_MHZ, PEAK_SOURCE = _measured_peaks()


def _median_loaded_mhz():
    try:
        return float(json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))["clocks_under_load"]["sm_mhz_median"])
    except (OSError, ValueError, KeyError, TypeError):
        return None


def measure_fp32_peak(dgf, torch, dev, seconds: float = 1.0):
    """FP32 FMA throughput of this GPU, measured with the library's probe (scalar FFMA
    and packed FP32x2 FMA over 8 resident blocks of 256 threads per SM), timed with
    CUDA events while nvidia-smi samples the SM clock; the tracking kernel's roofline
    denominator. Also scaled to the maximum and to the median loaded SM clock."""
    import ctypes
    lib = dgf.load()
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    blocks, threads, iters = sms * 8, 256, 20000
    out = torch.empty(blocks * threads, dtype=torch.float32, device=dev)
    stream = torch.cuda.current_stream(dev)
    s_ptr = ctypes.c_void_p(stream.cuda_stream)
    rec = {"sms": sms, "blocks": blocks, "threads": threads}
    for packed in (0, 1):
        def launch():
            rc = lib.dgf_fp32_probe(ctypes.c_void_p(out.data_ptr()), blocks, threads, iters, packed, s_ptr)
            if rc:
                raise RuntimeError(f"dgf_fp32_probe failed ({rc})")
        for _ in range(3):
            launch()
        torch.cuda.synchronize(dev)
        a = torch.cuda.Event(enable_timing=True)
        b = torch.cuda.Event(enable_timing=True)
        a.record(stream)
        launch()
        b.record(stream)
        b.synchronize()
        reps = max(3, int(seconds / max(a.elapsed_time(b) * 1e-3, 1e-4)))
        with ClockSampler(dev.index or 0) as clocks:
            a.record(stream)
            for _ in range(reps):
                launch()
            b.record(stream)
            b.synchronize()
        tflops = lib.dgf_fp32_probe_flops(blocks, threads, iters, packed) * reps / (a.elapsed_time(b) * 1e-3) / 1e12
        c = clocks.summary()
        key = "packed" if packed else "scalar"
        rec[key] = {"tflops": tflops, "clocks": c}
    best = max(rec["scalar"]["tflops"], rec["packed"]["tflops"])
    mhz = rec["packed"]["clocks"].get("sm_mhz") if rec["packed"]["tflops"] >= rec["scalar"]["tflops"] else \
        rec["scalar"]["clocks"].get("sm_mhz")
    rec["tflops"] = best
    rec["sm_mhz"] = mhz
    if mhz:
        rec["tflops_at_max_clock"] = best * SM_MAX_MHZ / mhz
        med = _median_loaded_mhz()
        if med:
            rec["tflops_at_median_loaded_clock"] = best * med / mhz
            rec["median_loaded_mhz"] = med
    return rec


def flops_model(radius: int, model: int):
    """Algorithmic FLOPs per Gauss-Newton iteration and per level set-up of one point.

    Per support sample and iteration: bilinear sample 9, residual 3 (model 4) or 1,
    Hampel weight 2, weighted regressors 3 or 2, normal-equation sums 16 + 8 (model 4)
    or 6 + 4; per iteration a 4x4 (55) or 2x2 (10) Cholesky solve. Per level set-up
    and sample: three bilinear samples 27 + gradient-matrix sums 6; plus 10.
    """
    n = (2 * radius + 1) ** 2
    per_sample = 9 + 3 + 2 + 3 + 16 + 8 if model == 4 else 9 + 1 + 2 + 2 + 6 + 4
    per_iter = per_sample * n + (55 if model == 4 else 10)
    per_setup = 33 * n + 10
    return per_iter, per_setup


def algorithmic_flops(iters: np.ndarray, status: np.ndarray, levels: int, radius: int, model: int) -> float:
    per_iter, per_setup = flops_model(radius, model)
    tracked = (status == 0) | (status == 4)
    setups = np.where(tracked, levels, 1).sum()  # lost points: only one set-up counted (lower bound)
    return float(iters.astype(np.int64).sum() * per_iter + setups * per_setup)


class ClockSampler:
    """nvidia-smi clock / throttle samples while the timed region runs."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index, self.rows, self.proc = index, [], None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except OSError:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.rows.append([x.strip() for x in line.split(",")])

    def __exit__(self, *exc):
        if self.proc:
            self.proc.terminate()
            self.proc.wait(timeout=5)
            self.t.join(timeout=5)

    def summary(self):
        if not self.rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        sm = [float(r[1]) for r in self.rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in self.rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in self.rows for i in range(4)
                          if len(r) > 5 + i and r[5 + i].lower() == "active"})
        return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(self.rows)}


TRAFFIC_SOURCES = ("rlof.cu", "track_index.cuh", "common.cuh", "batch.cuh")  # what the tracking kernel is compiled from


def tracking_sources_digest():
    h = hashlib.sha256()
    for name in TRAFFIC_SOURCES:
        h.update(open(os.path.join(ROOT, "paper_1901_09971_gb300", "csrc", name), "rb").read())
    return h.hexdigest()


def kernel_traffic():
    """DRAM bytes per rlof launch from the committed ncu summary, or None when a source
    of the kernel changed after the capture."""
    path = os.path.join(ROOT, "profiles", "rlof_track_traffic.json")
    try:
        rec = json.load(open(path))
        return rec["dram_bytes_per_launch"] if rec.get("sources_sha256") == tracking_sources_digest() else None
    except (OSError, ValueError, KeyError):
        return None


def run_batched(dgf, torch, dev, reps: int = 10):
    """The mixed-size batch workload: 64 pairs (640x480 .. 1280x720, step 2..6,
    window 8, 3 levels, 9x9 support) through one rlof_track_many call replayed from
    a CUDA graph; detection + pyramids are also timed alone (stages 1|2) for their
    HBM roofline. Under torchrun every rank tracks its longest-processing-time
    share of the batch (shard.ShardedBatch) and the time is the slowest rank's."""
    from paper_1901_09971_gb300 import shard
    specs = [(W, H, 8, st) for (W, H, st) in synth.make_batch_specs(64, 3000)]
    prm = dgf.RlofParams(levels=3, radius=4, max_iter=30, model=4)
    runner = shard.ShardedBatch(specs, prm, dev)
    frames = [synth.make_translation_pair(specs[i][0], specs[i][1], seed=3000 + i) for i in runner.indices]
    d1 = [torch.from_numpy(p.I1).to(dev) for p in frames]
    d2 = [torch.from_numpy(p.I2).to(dev) for p in frames]
    bt = runner.tracker
    bt.bind(d1, d2)
    with tempfile.TemporaryDirectory() as tmp:  # the launch shape, tuned on this batch
        tuned = bt.autotune(reps=3, path=os.path.join(tmp, "tune.json"))
    stream = torch.cuda.current_stream(dev)

    def timed(stages, reps):
        # the batch's frames and pyramids (about 1 GB) are far larger than L2, so
        # runs go back to back between two events (no flush, no host gap)
        for _ in range(3):
            bt.run(use_graph=True, stages=stages)
        torch.cuda.synchronize(dev)
        shard.barrier()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        for _ in range(reps):
            bt.run(use_graph=True, stages=stages)
        b.record(stream)
        b.synchronize()
        return shard.reduce_scalar(a.elapsed_time(b) / reps, "max", device=dev)

    t_all = timed(7, reps)
    t_dp = timed(1 | 2, 10 * reps)
    specs = runner.specs  # byte model below: this rank's share
    # algorithmic bytes of detection + both pyramids: frame 1 read twice, frame 2
    # once, key-points written, 3 FP32 planes of frame 1 and 1 of frame 2 per level,
    # each with its replicated border (DGF_PYR_APRON pixels on every side: the
    # clamped taps tracking reads without clamping), which the builder must write too
    A = dgf.PYR_APRON
    nbytes = nbytes_inner = 0
    for (W, H, win, step), n in zip(specs, bt.n):
        px = sum((W >> l) * (H >> l) for l in range(prm.levels))
        px_b = sum(((W >> l) + 2 * A) * ((H >> l) + 2 * A) for l in range(prm.levels))
        nbytes += 3 * W * H + 8 * n + 4 * 4 * px_b
        nbytes_inner += 3 * W * H + 8 * n + 4 * 4 * px
    nbytes = shard.reduce_scalar(nbytes, "sum", device=dev)
    nbytes_inner = shard.reduce_scalar(nbytes_inner, "sum", device=dev)
    npts = int(shard.reduce_scalar(sum(bt.n), "sum", device=dev))
    gbs = nbytes / (t_dp / 1e3) / 1e9
    return {"workload": "64 mixed pairs 640x480..1280x720, step 2..6, window 8, 3 levels, 9x9, model 4, FP32, "
                        "one rlof_track_many call replayed from a CUDA graph"
                        + (f", sharded over {runner.world} ranks by longest processing time" if runner.world > 1 else ""),
            "timing": f"{reps} (detect + pyramids alone: {10 * reps}) back-to-back runs between two CUDA events "
                      "(working set > L2, no flush)",
            "pairs": 64, "points": npts, "ms_per_batch": t_all, "points_per_s": npts / (t_all / 1e3),
            "pairs_per_s": 64 / (t_all / 1e3),
            "autotune": {"lanes_per_point": tuned["lanes"], "ms_per_batch_by_lanes": tuned["ms"]},
            "detect_pyramid": {"ms": t_dp, "algorithmic_bytes": nbytes, "achieved_gbs": gbs,
                               "frac_of_measured_hbm": gbs / (HBM_PEAK_GBS * runner.world),
                               "peak_gbs": HBM_PEAK_GBS * runner.world,
                               "peak_source": PEAK_SOURCE,
                               "bytes_without_border": nbytes_inner,
                               "frac_without_border": nbytes_inner / (t_dp / 1e3) / 1e9 / (HBM_PEAK_GBS * runner.world)}}


def _timed(torch, dev, fn, reps, flush):
    stream = torch.cuda.current_stream(dev)
    for _ in range(3):
        fn()
    torch.cuda.synchronize(dev)
    ms = []
    for k in range(reps):
        flush.fill_(k & 0xFF)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        fn()
        b.record(stream)
        b.synchronize()
        ms.append(a.elapsed_time(b))
    return float(np.median(ms))


def run_fp16(dgf, torch, dev, reps: int = 5):
    """FP16 pyramid storage against FP32 storage: 32 pairs at 1242x375 (translation
    flow, window 8, step 4, 3 levels, 9x9) through rlof_track_many."""
    pairs = [synth.make_pair(4, index=i) for i in range(32)]
    d1 = [torch.from_numpy(p.I1).to(dev) for p in pairs]
    d2 = [torch.from_numpy(p.I2).to(dev) for p in pairs]
    specs = [(pairs[0].W, pairs[0].H, 8, 4)] * 32
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=dev)
    out = {"workload": "32 pairs 1242x375, translation flow, window 8, step 4, 3 levels, 9x9, model 4"}
    for name, storage in (("f32", dgf.F32), ("f16", dgf.F16)):
        bt = dgf.BatchTracker(specs, dgf.RlofParams(levels=3, radius=4, max_iter=30, model=4, storage=storage), dev)
        t = _timed(torch, dev, lambda: bt.run(d1, d2, use_graph=True), reps, flush)
        out[name] = {"ms_per_batch": t, "points_per_s": sum(bt.n) / (t / 1e3)}
    out["f16_speedup"] = out["f32"]["ms_per_batch"] / out["f16"]["ms_per_batch"]
    return out


def run_adjoint(dgf, torch, dev, reps: int = 5):
    """Forward + implicit adjoint of tracking for 8 pairs at 1242x375 (step 4, 3
    levels, 9x9, model 4), loss = sum of w . flow with w ~ N(0, 1) per point."""
    pairs = [synth.make_pair(5, index=i) for i in range(8)]
    prm = dgf.RlofParams(levels=3, radius=4, max_iter=30, model=4)
    frames = [(torch.from_numpy(p.I1).float().to(dev), torch.from_numpy(p.I2).float().to(dev)) for p in pairs]
    pts = [dgf.detect(torch.from_numpy(p.I1).to(dev), 8, 4) for p in pairs]
    ws = [torch.randn(pt.shape, device=dev) for pt in pts]
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=dev)

    def step():
        for (f1, f2), pt, w in zip(frames, pts, ws):
            a = f1.detach().requires_grad_(True)
            b = f2.detach().requires_grad_(True)
            flow, _ = dgf.RLOFTrack.apply(a, b, pt, prm)
            (flow * w).sum().backward()

    t = _timed(torch, dev, step, reps, flush)
    return {"workload": "8 pairs 1242x375, step 4, 3 levels, 9x9, model 4: forward + implicit adjoint (torch autograd)",
            "ms_per_8_pairs": t, "pairs_per_s": 8 / (t / 1e3)}


def hbm_context(W: int, H: int, n: int, ms_per_step: float):
    """The whole step's HBM fraction under two byte models, reported beside the FP32
    fraction of tracking (the step is ALU-bound, so both are small): I/O only (both
    frames in; points, flow and status out) and with the pyramid materialised (4
    FP32 planes over the levels, their replicated borders included, written once
    and read once, the points re-read)."""
    A = 12  # the pyramid planes' replicated border (DGF_PYR_APRON)
    px = sum(((W >> l) + 2 * A) * ((H >> l) + 2 * A) for l in range(WORKLOAD["levels"]))
    io = 2 * W * H + n * (8 + 8 + 1)
    mat = io + 2 * 4 * 4 * px + 8 * n
    gbs = lambda b: b / (ms_per_step / 1e3) / 1e9
    return {"io_only_bytes": io, "materialised_bytes": mat, "io_only_frac": gbs(io) / HBM_PEAK_GBS,
            "materialised_frac": gbs(mat) / HBM_PEAK_GBS, "peak_gbs": HBM_PEAK_GBS,
            "note": "tracking is FP32-ALU bound (roofline above); the HBM traffic of a step is a few MB"}


def run_small_pair(dgf, torch, dev, reps: int = 50):
    """The 256x128 translation pair (window 8, step 4, 3 levels, 9x9): one step
    (detection, both pyramids, tracking) on device frames, as one replayed CUDA graph
    of the batched entry, and as four separate launches (PairTracker)."""
    p = synth.make_pair(1)
    prm = dgf.RlofParams(levels=p.levels, radius=p.radius, max_iter=p.max_iter, model=4)
    f1, f2 = torch.from_numpy(p.I1).to(dev), torch.from_numpy(p.I2).to(dev)
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=dev)
    bt = dgf.BatchTracker([(p.W, p.H, p.win, p.step)], prm, dev)
    bt.bind([f1], [f2])
    t = _timed(torch, dev, lambda: bt.run(use_graph=True), reps, flush)
    tr = dgf.PairTracker(p.W, p.H, p.win, p.step, prm, dev)
    t4 = _timed(torch, dev, lambda: tr.run(f1, f2), reps, flush)
    n = bt.n[0]
    return {"workload": f"256x128 translation pair, window 8, step 4 ({n} points), 3 levels, 9x9, model 4, FP32",
            "ms_per_step": t, "points_per_s": n / (t / 1e3), "pairs_per_s": 1e3 / t,
            "ms_per_step_four_launches": t4}


def run_gm_prior(dgf, torch, dev, pair, reps: int = 20):
    """The global-motion prior on the 1242x375 pair: plain tracking against
    rlof_track_gm (sparse first pass every 4th point, affine fit, main pass), both
    on device-resident pyramids; quality = fraction of non-occluded points tracked
    (TRACKED) within 2 px of the ground-truth flow."""
    prm = dgf.RlofParams(levels=WORKLOAD["levels"], radius=WORKLOAD["radius"], max_iter=WORKLOAD["max_iter"],
                         model=WORKLOAD["model"])
    gm = dgf.GmParams(extra_levels=0)  # 5 levels already reach the frame's coarsest usable size
    f1 = torch.from_numpy(pair.I1).to(dev)
    p1 = dgf.build_pyramid(f1, prm.levels, prm.storage, True)
    p2 = dgf.build_pyramid(torch.from_numpy(pair.I2).to(dev), prm.levels, prm.storage, False)
    pts = dgf.detect(f1, WORKLOAD["win"], WORKLOAD["step"])
    n = pts.shape[0]
    ws = torch.zeros(dgf.gm_workspace_bytes(n, gm), dtype=torch.uint8, device=dev)
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=dev)
    plain = lambda: dgf.track(p1, p2, pair.W, pair.H, pts, prm)
    prior = lambda: dgf.track_gm(p1, p2, pair.W, pair.H, prm.levels, pts, prm, gm, workspace=ws)
    t_plain = _timed(torch, dev, plain, reps, flush)
    t_gm = _timed(torch, dev, prior, reps, flush)
    P = pts.cpu().numpy()
    ix = np.clip(np.rint(P[:, 0]), 0, pair.W - 1).astype(int)
    iy = np.clip(np.rint(P[:, 1]), 0, pair.H - 1).astype(int)
    gt = pair.flow_gt[iy, ix].astype(np.float64)
    vis = ~pair.occluded[iy, ix]

    def good(flow, status):
        f, st = flow.cpu().numpy(), status.cpu().numpy()
        return float(np.mean(((st == dgf.TRACKED) & (np.hypot(*(f - gt).T) < 2.0))[vis]))

    fp, sp = plain()
    fg, sg, a, made = prior()
    return {"workload": "1242x375 driving-scene pair, 5 levels, 11x11: plain tracking vs the global-motion prior "
                        "(first pass every 4th point, affine Tukey IRLS, main pass from the prior)",
            "plain_ms": t_plain, "gm_ms": t_gm, "gm_points_per_s": n / (t_gm / 1e3),
            "within_2px_of_truth": {"plain": good(fp, sp), "gm": good(fg, sg)},
            "affine": [float(v) for v in a.cpu().numpy()], "fitted": bool(int(made.item()))}


def run_cross_support(dgf, torch, dev, pair, reps: int = 20, tau: float = 20.0):
    """The adaptive cross-based support on the 1242x375 pair (rectangles moving over
    the radially expanding background: motion boundaries): square vs cross support,
    time and fraction of non-occluded points tracked within 2 px of the truth."""
    base = dict(levels=WORKLOAD["levels"], radius=WORKLOAD["radius"], max_iter=WORKLOAD["max_iter"],
                model=WORKLOAD["model"])
    f1 = torch.from_numpy(pair.I1).to(dev)
    p1 = dgf.build_pyramid(f1, base["levels"], dgf.F32, True)
    p2 = dgf.build_pyramid(torch.from_numpy(pair.I2).to(dev), base["levels"], dgf.F32, False)
    pts = dgf.detect(f1, WORKLOAD["win"], WORKLOAD["step"])
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=dev)
    P = pts.cpu().numpy()
    ix = np.clip(np.rint(P[:, 0]), 0, pair.W - 1).astype(int)
    iy = np.clip(np.rint(P[:, 1]), 0, pair.H - 1).astype(int)
    gt = pair.flow_gt[iy, ix].astype(np.float64)
    vis = ~pair.occluded[iy, ix]
    out = {"workload": f"1242x375 driving-scene pair, 5 levels, 11x11: square support vs cross support (tau {tau})"}
    for name, prm in (("square", dgf.RlofParams(**base)), ("cross", dgf.RlofParams(**base, cross_tau=tau))):
        fn = lambda: dgf.track(p1, p2, pair.W, pair.H, pts, prm)
        t = _timed(torch, dev, fn, reps, flush)
        f, st = fn()
        f, st = f.cpu().numpy(), st.cpu().numpy()
        good = float(np.mean(((st == dgf.TRACKED) & (np.hypot(*(f - gt).T) < 2.0))[vis]))
        out[name] = {"ms": t, "within_2px_of_truth": good}
    return out


def run_fb_filter(dgf, torch, dev, pair, reps: int = 20, fb_max: float = 1.0):
    """The forward-backward filter on the 1242x375 pair: its time against one tracking
    pass, and how often it rejects forward-tracked points that are wrong (more than
    2 px from the truth) against points that are right."""
    prm = dgf.RlofParams(levels=WORKLOAD["levels"], radius=WORKLOAD["radius"], max_iter=WORKLOAD["max_iter"],
                         model=WORKLOAD["model"])
    f1 = torch.from_numpy(pair.I1).to(dev)
    p1 = dgf.build_pyramid(f1, prm.levels, dgf.F32, True)
    p2 = dgf.build_pyramid(torch.from_numpy(pair.I2).to(dev), prm.levels, dgf.F32, True)
    pts = dgf.detect(f1, WORKLOAD["win"], WORKLOAD["step"])
    ws = torch.empty(int(dgf.load().dgf_fb_workspace(pts.shape[0])), dtype=torch.uint8, device=dev)
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=dev)
    t_one = _timed(torch, dev, lambda: dgf.track(p1, p2, pair.W, pair.H, pts, prm), reps, flush)
    fb = lambda: dgf.track_fb(p1, p2, pair.W, pair.H, pts, prm, fb_max, workspace=ws)
    t_fb = _timed(torch, dev, fb, reps, flush)
    f, st, err = (x.cpu().numpy() for x in fb())
    P = pts.cpu().numpy()
    ix = np.clip(np.rint(P[:, 0]), 0, pair.W - 1).astype(int)
    iy = np.clip(np.rint(P[:, 1]), 0, pair.H - 1).astype(int)
    wrong = np.hypot(*(f - pair.flow_gt[iy, ix]).T) > 2.0
    fwd = np.isin(st, [dgf.TRACKED, dgf.MAXITER, dgf.FB_REJECTED])
    rej = st == dgf.FB_REJECTED
    return {"workload": f"1242x375 driving-scene pair, 5 levels, 11x11, fb_max {fb_max} px",
            "one_pass_ms": t_one, "fb_ms": t_fb,
            "rejected_of_wrong": float(np.mean(rej[fwd & wrong])), "rejected_of_right": float(np.mean(rej[fwd & ~wrong]))}


def run_epic(dgf, torch, dev, pair, reps: int = 20):
    """EPIC interpolation of the 1242x375 pair's sparse flow into a dense field: the
    time of one epic_interpolate call (k = 128) and the dense end-point error on
    non-occluded pixels for three sparse inputs: plain tracking, tracking with the
    global-motion prior, and the ground truth at the key-points (interpolation
    alone)."""
    prm = dgf.RlofParams(levels=WORKLOAD["levels"], radius=WORKLOAD["radius"], max_iter=WORKLOAD["max_iter"],
                         model=WORKLOAD["model"])
    f1 = torch.from_numpy(pair.I1).to(dev)
    p1 = dgf.build_pyramid(f1, prm.levels, dgf.F32, True)
    p2 = dgf.build_pyramid(torch.from_numpy(pair.I2).to(dev), prm.levels, dgf.F32, False)
    pts = dgf.detect(f1, WORKLOAD["win"], WORKLOAD["step"])
    n = pts.shape[0]
    flow, st = dgf.track(p1, p2, pair.W, pair.H, pts, prm)
    gm = dgf.GmParams(extra_levels=0)  # as in the gm_prior section
    gflow, gst = dgf.track_gm(p1, p2, pair.W, pair.H, prm.levels, pts, prm, gm)[:2]
    P = pts.cpu().numpy()
    ix = np.clip(np.rint(P[:, 0]), 0, pair.W - 1).astype(int)
    iy = np.clip(np.rint(P[:, 1]), 0, pair.H - 1).astype(int)
    truth = torch.from_numpy(np.ascontiguousarray(pair.flow_gt[iy, ix], dtype=np.float32)).to(dev)
    tst = torch.from_numpy(np.where(pair.occluded[iy, ix], dgf.OOB, dgf.TRACKED).astype(np.uint8)).to(dev)
    ep = dgf.EpicParams()
    ws = torch.empty(dgf.epic_workspace_bytes(pair.W, pair.H, n), dtype=torch.uint8, device=dev)
    dense = torch.empty((pair.H, pair.W, 2), dtype=torch.float32, device=dev)
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=dev)
    t = _timed(torch, dev, lambda: dgf.epic_interpolate(f1, pts, flow, st, ep, workspace=ws), reps, flush)
    vis = ~pair.occluded
    out = {"workload": f"1242x375 driving-scene pair, {n} key-points, k {ep.k}, affine fits", "ms": t}
    for name, (fl, ss) in {"plain_tracks": (flow, st), "gm_prior_tracks": (gflow, gst),
                           "truth_at_keypoints": (truth, tst)}.items():
        dense = dgf.epic_interpolate(f1, pts, fl.contiguous(), ss.contiguous(), ep, workspace=ws).cpu().numpy()
        e = np.hypot(*(dense.astype(np.float64) - pair.flow_gt).transpose(2, 0, 1))[vis]
        out[name] = {"epe_noc_px": float(e.mean()), "fl_noc_over_3px": float(np.mean(e > 3.0))}
    return out


def run_dense_pipeline(dgf, torch, dev, pair, reps: int = 20):
    """The whole DeGraF-Flow method on the 1242x375 pair: DeGraF points, pyramids,
    tracking with the global-motion prior (RLOF(IM-GM)) and EPIC interpolation into a
    dense field, one DenseFlow run per pair; dense EPE on non-occluded pixels."""
    prm = dgf.RlofParams(levels=WORKLOAD["levels"], radius=WORKLOAD["radius"], max_iter=WORKLOAD["max_iter"],
                         model=WORKLOAD["model"])
    df = dgf.DenseFlow(pair.W, pair.H, WORKLOAD["win"], WORKLOAD["step"], prm, gm=dgf.GmParams(extra_levels=0),
                       device=dev)
    f1 = torch.from_numpy(pair.I1).to(dev)
    f2 = torch.from_numpy(pair.I2).to(dev)
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=dev)
    t_eager = _timed(torch, dev, lambda: df.run(f1, f2), reps, flush)
    # a run waits on nothing on the host, so it is captured once into a CUDA graph and
    # replayed (no launch gaps between its 20-odd kernels)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        dense_g = df.run(f1, f2)[0]
    t = _timed(torch, dev, g.replay, reps, flush)
    dense = dense_g.cpu().numpy().astype(np.float64)
    e = np.hypot(*(dense - pair.flow_gt).transpose(2, 0, 1))[~pair.occluded]
    return {"workload": "1242x375 driving-scene pair: DeGraF w7 s3 (50,676 points), pyramids, RLOF 5 levels 11x11 "
                        "with the global-motion prior, EPIC k 128 into a dense field, one captured CUDA graph "
                        "replayed per pair",
            "ms_per_pair": t, "pairs_per_s": 1e3 / t, "ms_per_pair_eager": t_eager, "epe_noc_px": float(e.mean()),
            "fl_noc_over_3px": float(np.mean(e > 3.0)),
            "paper_context": "the paper's C++ pipeline (detection + RLOF + EPIC): 3.2 s per KITTI pair on 4 CPU cores"}


def cpu_baseline(pair, reps: int = 2):
    """The FP64 oracle as it stands, on this host's cores, over the full pair."""
    import oracle
    prm = oracle.RlofParams(levels=WORKLOAD["levels"], radius=WORKLOAD["radius"],
                            max_iter=WORKLOAD["max_iter"], model=WORKLOAD["model"])
    threads = oracle.max_threads()
    t0 = time.perf_counter()
    n = 0
    for _ in range(reps):
        pts, _, _ = oracle.degraf_detect(pair.I1, WORKLOAD["win"], WORKLOAD["win"], WORKLOAD["step"])
        oracle.rlof_track(pair.I1, pair.I2, pts, prm)
        n += pts.shape[0]
    dt = time.perf_counter() - t0
    return {"value": n / dt, "unit": "points/s", "cores": threads, "kind": "oracle",
            "sample": f"full 1242x375 pair ({n // reps} points, detection + pyramids + tracking) x {reps}, "
                      f"{dt:.1f} s wall"}


def oracle_next_rows(dgf, torch, dev, pair):
    """The FP64 oracle of each extension timed on this host beside its GPU section
    (part of the CPU baseline leg), on the same 1242x375 pair: the global-motion
    prior, the cross-based support (tau 20), the forward-backward filter (1 px), and
    EPIC (k 128) on the GPU's plain tracks. One run each, wall time on all cores."""
    import oracle
    prm = oracle.RlofParams(levels=WORKLOAD["levels"], radius=WORKLOAD["radius"], max_iter=WORKLOAD["max_iter"],
                            model=WORKLOAD["model"])
    f1 = torch.from_numpy(pair.I1).to(dev)
    pts_d = dgf.detect(f1, WORKLOAD["win"], WORKLOAD["step"])
    pts = pts_d.cpu().numpy().astype(np.float64)
    out = {}

    def timed(name, fn):
        t0 = time.perf_counter()
        fn()
        out[name] = {"oracle_ms": 1e3 * (time.perf_counter() - t0), "cores": oracle.max_threads(), "kind": "oracle"}

    timed("gm_prior", lambda: oracle.rlof_track_gm(pair.I1, pair.I2, pts, prm, extra_levels=0))
    timed("cross_support", lambda: oracle.rlof_track(pair.I1, pair.I2, pts,
                                                     oracle.RlofParams(**{**prm.__dict__, "cross_tau": 20.0})))
    timed("fb_filter", lambda: oracle.rlof_track_fb(pair.I1, pair.I2, pts, prm, 1.0))
    gp = dgf.RlofParams(levels=prm.levels, radius=prm.radius, max_iter=prm.max_iter, model=prm.model)
    p1 = dgf.build_pyramid(f1, gp.levels, dgf.F32, True)
    p2 = dgf.build_pyramid(torch.from_numpy(pair.I2).to(dev), gp.levels, dgf.F32, False)
    flow, status = dgf.track(p1, p2, pair.W, pair.H, pts_d, gp)
    fl, st = flow.cpu().numpy().astype(np.float64), status.cpu().numpy()
    timed("epic", lambda: oracle.epic_interpolate(pair.I1, pts, fl, st, oracle.EpicParams()))
    return out


def oracle_epe(dgf, torch, dev, pair):
    """End-point error of the GPU path against the FP64 oracle (part of the CPU
    baseline leg: the oracle runs on this host), per workload, on the GPU's own
    key-points: the 1242x375 pair in full, the 256x128 pair, two pairs of the mixed
    batch, and two 1242x375 translation pairs with FP32 and FP16 pyramid storage.
    EPE over the points both sides tracked to convergence (TRACKED), with the
    status agreement over all points."""
    import oracle

    def compare(I1, I2, win, step, levels, radius, storages=(("f32", None),)):
        H, W = I1.shape
        f1 = torch.from_numpy(I1).to(dev)
        pts = dgf.detect(f1, win, step)
        P = pts.cpu().numpy().astype(np.float64)
        fo, so, _, _ = oracle.rlof_track(I1, I2, P, oracle.RlofParams(levels=levels, radius=radius, max_iter=30,
                                                                      model=4))
        out = {}
        for name, storage in storages:
            storage = dgf.F32 if storage is None else storage
            prm = dgf.RlofParams(levels=levels, radius=radius, max_iter=30, model=4, storage=storage)
            p1 = dgf.build_pyramid(f1, levels, storage, True)
            p2 = dgf.build_pyramid(torch.from_numpy(I2).to(dev), levels, storage, False)
            fg, sg = dgf.track(p1, p2, W, H, pts, prm)
            fg, sg = fg.cpu().numpy().astype(np.float64), sg.cpu().numpy()
            both = (sg == dgf.TRACKED) & (so == dgf.TRACKED)
            e = np.hypot(*(fg - fo)[both].T)
            out[name] = {"points": int(len(sg)), "both_tracked": int(both.sum()), "epe_mean_px": float(e.mean()),
                         "epe_p99_px": float(np.percentile(e, 99)), "epe_max_px": float(e.max()),
                         "within_1e-2_px": float(np.mean(e <= 1e-2)), "status_agreement": float(np.mean(sg == so))}
        return out if len(storages) > 1 else out["f32"]

    res = {"definition": "unsquared end-point difference GPU vs FP64 oracle on points TRACKED by both; "
                         "status agreement over all points"}
    res["driving_scene_1242x375"] = compare(pair.I1, pair.I2, WORKLOAD["win"], WORKLOAD["step"], WORKLOAD["levels"],
                                            WORKLOAD["radius"])
    p1 = synth.make_pair(1)
    res["translation_256x128"] = compare(p1.I1, p1.I2, p1.win, p1.step, p1.levels, p1.radius)
    specs = synth.make_batch_specs(64, 3000)
    for i in range(2):
        W, H, st = specs[i]
        fr = synth.make_translation_pair(W, H, seed=3000 + i)
        res[f"batch_pair_{i}_{W}x{H}_step{st}"] = compare(fr.I1, fr.I2, 8, st, 3, 4)
    for i in range(2):
        q = synth.make_pair(4, index=i)
        res[f"storage_pair_{i}_1242x375"] = compare(q.I1, q.I2, 8, 4, 3, 4, (("f32", dgf.F32), ("f16", dgf.F16)))
    return res


REF_BUDGET_S = 90.0  # host wall time a whole reference run (warm-up + timed steps) aims for


def run_reference(args, rank: int, world: int):
    """The FP64 oracle on the host cores, on the bench's workload: per step, detection
    and pyramids of the full 1242x375 pair and tracking of an evenly strided sample of
    its key-points, sized from a measured tracking rate so that the whole run stays
    near REF_BUDGET_S whatever --steps and --warmup are."""
    if rank != 0:
        return
    pair = synth.make_pair(2)
    import oracle
    prm = oracle.RlofParams(levels=WORKLOAD["levels"], radius=WORKLOAD["radius"],
                            max_iter=WORKLOAD["max_iter"], model=WORKLOAD["model"])
    pts_all, _, _ = oracle.degraf_detect(pair.I1, WORKLOAD["win"], WORKLOAD["win"], WORKLOAD["step"])
    n_all = pts_all.shape[0]
    probe = pts_all[::max(1, n_all // 4096)]
    t0 = time.perf_counter()
    oracle.rlof_track(pair.I1, pair.I2, probe, prm)
    rate = probe.shape[0] / (time.perf_counter() - t0)
    per_step = min(n_all, max(512, int(REF_BUDGET_S * rate / (args.steps + args.warmup))))
    stride = max(1, -(-n_all // per_step))

    def step():
        pts, _, _ = oracle.degraf_detect(pair.I1, WORKLOAD["win"], WORKLOAD["win"], WORKLOAD["step"])
        sample = pts[::stride]
        oracle.rlof_track(pair.I1, pair.I2, sample, prm)
        return sample.shape[0]

    for _ in range(args.warmup):
        step()
    t0 = time.perf_counter()
    n = sum(step() for _ in range(args.steps))
    dt = time.perf_counter() - t0
    value = n / dt
    cores = oracle.max_threads()
    line = {"metric": METRIC, "value": value, "unit": "points/s", "n_gpus": args.gpus, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": 1e3 * dt / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "impl": "reference", "config": {k: v for k, v in WORKLOAD.items()},
            "cpu_baseline": {"value": value, "unit": "points/s", "cores": cores, "kind": "oracle",
                             "sample": f"per step: detection of the full 1242x375 pair and tracking (pyramids "
                                       f"included) of {'all' if stride == 1 else f'every {stride}th'} of its "
                                       f"{n_all} key-points ({n} points over {args.steps} timed steps, {dt:.1f} s)"},
            "e2e": {"value": value, "unit": "points/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
            "gpu_launches": 0}
    print(json.dumps(line), flush=True)


def run_cuda(args, rank: int, world: int, local_rank: int):
    import torch
    import paper_1901_09971_gb300 as dgf
    from paper_1901_09971_gb300 import shard

    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    if args.batched_only:  # profiling aid: the 64-pair batch section alone, no bench line
        if rank == 0:
            print(json.dumps({"batched": run_batched(dgf, torch, dev)}), flush=True)
        return
    if args.adjoint_only:  # profiling aid: the adjoint section alone, no bench line
        if rank == 0:
            print(json.dumps({"adjoint": run_adjoint(dgf, torch, dev, reps=args.steps)}), flush=True)
        return
    if args.epic_only:  # profiling aid: the EPIC section alone, no bench line
        if rank == 0:
            print(json.dumps({"epic": run_epic(dgf, torch, dev, synth.make_pair(2), reps=args.steps)}), flush=True)
        return
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)
    # the step's pairs: one driving-scene pair per rank, split by the same
    # longest-processing-time partition as any batch (equal costs: pair k on rank k)
    step_pairs = [(1242, 375, WORKLOAD["win"], WORKLOAD["step"])] * world
    (mine,), _ = shard.shard_specs(step_pairs, WORKLOAD["levels"], WORKLOAD["radius"], rank, world)
    pair = synth.make_pair(2, index=mine)
    W, H = pair.W, pair.H
    prm = dgf.RlofParams(levels=WORKLOAD["levels"], radius=WORKLOAD["radius"], max_iter=WORKLOAD["max_iter"],
                         model=WORKLOAD["model"])
    # the library's batched entry for this one pair: detection beside both frames'
    # pyramids (one launch) in a replayed CUDA graph, then tracking (one launch)
    spec = [(W, H, WORKLOAD["win"], WORKLOAD["step"])]
    tr = dgf.BatchTracker(spec, prm, dev)
    if args.lanes:
        tr.lanes = args.lanes
    f1 = torch.from_numpy(pair.I1).to(dev)
    f2 = torch.from_numpy(pair.I2).to(dev)
    tr.bind([f1], [f2])
    flush = torch.empty(L2_FLUSH_BYTES, dtype=torch.uint8, device=dev)
    stream = torch.cuda.current_stream(dev)
    from paper_1901_09971_gb300 import _abi

    def one_step(ev):
        ev[0].record(stream)
        tr.run(use_graph=True, stages=_abi.STAGE_DETECT | _abi.STAGE_PYRAMID)
        ev[1].record(stream)
        tr.run(use_graph=False, stages=_abi.STAGE_TRACK)
        ev[2].record(stream)

    for _ in range(args.warmup):
        flush.fill_(1)
        one_step([torch.cuda.Event(enable_timing=True) for _ in range(3)])
    torch.cuda.synchronize(dev)
    evs = [[torch.cuda.Event(enable_timing=True) for _ in range(3)] for _ in range(args.steps)]
    with ClockSampler(local_rank) as clocks:
        if dist:
            dist.barrier()
        torch.cuda.synchronize(dev)
        for k in range(args.steps):
            flush.fill_(k & 0xFF)  # evict L2 between steps (outside the timed events)
            one_step(evs[k])
        torch.cuda.synchronize(dev)
        if dist:
            dist.barrier()
    step_ms = np.array([e[0].elapsed_time(e[2]) for e in evs])
    rlof_ms = np.array([e[1].elapsed_time(e[2]) for e in evs])
    total_s = step_ms.sum() / 1e3
    total_s = shard.reduce_scalar(total_s, "max", device=dev)  # slowest rank
    n_pts = tr.n[0]
    value = world * n_pts * args.steps / total_s

    # dominant kernel: RLOF tracking, algorithmic FLOPs of the last step's trajectories
    iters = tr.iters[0].cpu().numpy()
    status = tr.status[0].cpu().numpy()
    flops = algorithmic_flops(iters, status, prm.levels, prm.radius, prm.model)
    achieved = flops / (rlof_ms.mean() / 1e3) / 1e12
    fp32 = measure_fp32_peak(dgf, torch, dev)

    # end to end through the public API: pinned host frames in, host results out
    # (HostPairTracker.run: host-to-device copies, the pair, device-to-host copies
    # and the wait for them)
    h1 = torch.from_numpy(pair.I1).pin_memory()
    h2 = torch.from_numpy(pair.I2).pin_memory()
    o_pts = torch.empty((n_pts, 2), dtype=torch.float32).pin_memory()
    o_flow = torch.empty((n_pts, 2), dtype=torch.float32).pin_memory()
    o_status = torch.empty(n_pts, dtype=torch.uint8).pin_memory()
    te = dgf.HostPairTracker(W, H, WORKLOAD["win"], WORKLOAD["step"], prm, dev, lanes=tr.lanes)

    def e2e_step():
        te.run(h1, h2, out=(o_pts, o_flow, o_status))

    for _ in range(3):
        e2e_step()
    torch.cuda.synchronize(dev)
    e_ms = []
    for k in range(args.steps):
        flush.fill_(k & 0xFF)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        e2e_step()
        b.record(stream)
        b.synchronize()
        e_ms.append(a.elapsed_time(b))
    e2e_s = sum(e_ms) / 1e3
    e2e_s = shard.reduce_scalar(e2e_s, "max", device=dev)
    e2e_value = world * n_pts * args.steps / e2e_s

    # the 64-pair batch, every rank tracking its share (all ranks take part)
    batched = None if args.no_batched else run_batched(dgf, torch, dev)

    if rank == 0:
        line = {"metric": METRIC, "value": value, "unit": "points/s", "n_gpus": world, "steps": args.steps,
                "warmup": args.warmup, "ms_per_step": 1e3 * total_s / args.steps, "higher_is_better": True,
                "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
                "config": dict(WORKLOAD, points_per_pair=n_pts, l2="flushed between steps (256 MiB write)",
                               parallelism=f"pairs sharded over {world} ranks (one pair each per step)"
                               if world > 1 else "single GPU"),
                "pairs_per_s": world * args.steps / total_s,
                "rlof_ms": float(rlof_ms.mean()), "detect_pyramid_ms": float((step_ms - rlof_ms).mean()),
                "tracked_fraction": float(np.mean((status == 0) | (status == 4))),
                "roofline": {"bound": "alu", "achieved": achieved, "peak": fp32["tflops"], "unit": "TFLOP/s",
                             "frac": achieved / fp32["tflops"], "traffic": kernel_traffic(),
                             "peak_basis": f"measured: FP32 FMA probe (dgf_fp32_probe, the faster of scalar and "
                                           f"packed FMA) on {fp32['sms']} SMs at a median {fp32['sm_mhz']} MHz, "
                                           f"CUDA events",
                             "kernel": "rlof_kernel", "flops_per_launch": flops,
                             "flops_basis": "every iteration counted as a full step; a step whose residuals all "
                                            "have weight 1 (18% of this pair's) does about two thirds of it"},
                "fp32_peak": fp32,
                "e2e": {"value": e2e_value, "unit": "points/s", "h2d_bytes_per_step": 2 * W * H,
                        "d2h_bytes_per_step": n_pts * (8 + 8 + 1)},
                "gpu_launches": 3 * args.steps,
                "clocks": clocks.summary()}
        line["hbm_context"] = hbm_context(W, H, n_pts, 1e3 * total_s / args.steps)
        if batched is not None:
            line["batched"] = batched
            dp = batched["detect_pyramid"]
            # the HBM-bound stages' roofline beside the dominant kernel's
            line["roofline"]["secondary"] = [{
                "kernel": "degraf_detect_kernel + pyramid_kernel, 64 mixed pairs (one graph replay)",
                "bound": "hbm", "achieved": dp["achieved_gbs"], "peak": dp["peak_gbs"], "unit": "GB/s",
                "frac": dp["frac_of_measured_hbm"], "ms": dp["ms"], "bytes": dp["algorithmic_bytes"]}]
        if not args.no_batched:
            line["small_pair"] = run_small_pair(dgf, torch, dev)
            line["fp16_storage"] = run_fp16(dgf, torch, dev)
            line["adjoint"] = run_adjoint(dgf, torch, dev)
            line["gm_prior"] = run_gm_prior(dgf, torch, dev, pair)
            line["cross_support"] = run_cross_support(dgf, torch, dev, pair)
            line["fb_filter"] = run_fb_filter(dgf, torch, dev, pair)
            line["epic"] = run_epic(dgf, torch, dev, pair)
            line["dense_pipeline"] = run_dense_pipeline(dgf, torch, dev, pair)
        if world == 1 and not args.no_cpu_baseline:
            line["cpu_baseline"] = cpu_baseline(pair)
            line["epe_vs_oracle"] = oracle_epe(dgf, torch, dev, pair)
            if not args.no_batched:
                for name, rec in oracle_next_rows(dgf, torch, dev, pair).items():
                    line[name]["oracle"] = rec
        print(json.dumps(line), flush=True)
    if dist:
        dist.destroy_process_group()


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", choices=["cuda", "reference"], default="cuda")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-batched", action="store_true",
                    help="skip every section after the main step (small pair, batch, FP16 storage, adjoint, "
                         "global-motion prior, cross support, forward-backward filter, EPIC, dense pipeline)")
    ap.add_argument("--lanes", type=int, default=0, help="lanes per tracked point (0 = automatic)")
    ap.add_argument("--batched-only", action="store_true",
                    help="run only the 64-pair batch section and print its JSON (for profiling)")
    ap.add_argument("--adjoint-only", action="store_true",
                    help="run only the adjoint section (--steps timed runs) and print its JSON (for profiling)")
    ap.add_argument("--epic-only", action="store_true",
                    help="run only the EPIC section (--steps timed calls) and print its JSON (for profiling)")
    args = ap.parse_args()
    args.warmup = max(args.warmup, 3)
    rank = int(os.environ.get("RANK", 0))
    world = int(os.environ.get("WORLD_SIZE", 1))
    local_rank = int(os.environ.get("LOCAL_RANK", 0))
    if args.impl == "reference":
        run_reference(args, rank, world)
    else:
        run_cuda(args, rank, world, local_rank)


if __name__ == "__main__":
    main()
