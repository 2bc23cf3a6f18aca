#!/usr/bin/env python
"""Throughput benchmark of the FUSE-Flow per-frame fusion path on GB300.

Workload: the 8-camera 1280x720 rig (uint16 depth in mm, float32 confidence, uint8 RGB),
300 frames per step as in the 300-frame sequence of that rig, fused 4 frames per batched
launch (every frame kernel launched once for the 4 frames) replayed from captured CUDA
graphs.  A pool of distinct seeded frames (larger than L2) is cycled, so every frame is
re-read from HBM.  The same frames one per fuse call are reported beside it.

Prints ONE JSON line on rank 0.  ``--impl reference`` times the FP64 CPU oracle (the only
reference implementation of the method) on the host cores instead.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "depth px/s and frames/s at 8x1280x720 views; p50/p99 latency, served vs plain"
KERNELS_PER_FRAME = 5      # count, levels, weigh, sum, emit (top-k: assign and reduce in place of weigh and sum)
CELL_OUT_BYTES = 44        # pos 12 + rgb 12 + weight 4 + count 4 + rep 4 + key 8
SERVE_MAX_SLOTS = 2        # frames of one served rig in flight at most (slots asked per rig)


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=30)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--frames-per-step", type=int, default=300)
    ap.add_argument("--pool", type=int, default=8, help="distinct frames cycled (> L2 in total)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--e2e-frames", type=int, default=256)
    ap.add_argument("--slots", type=int, default=4,
                    help="frames in flight on separate streams for the batched line")
    ap.add_argument("--serve-seconds", type=float, default=60.0,
                    help="length of the Poisson arrival trace of the served/plain comparison")
    ap.add_argument("--no-serving", action="store_true")
    ap.add_argument("--serve-slots", type=int, default=SERVE_MAX_SLOTS,
                    help="frames of one served rig in flight at most (slots asked per rig)")
    ap.add_argument("--serve-max-inflight", type=int, default=0,
                    help="frames on the device at once in the served replay (0: every free slot)")
    ap.add_argument("--no-autotune", action="store_true",
                    help="keep fuseflow_create's launch geometry instead of the autotuner's")
    return ap.parse_args()


def dist_env():
    return (int(os.environ.get("RANK", "0")), int(os.environ.get("WORLD_SIZE", "1")),
            int(os.environ.get("LOCAL_RANK", "0")))


def load_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


# ----------------------------------------------------------------------------- clocks
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")
    NAMES = ("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.tmp = None

    def start(self):
        try:
            self.tmp = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "50"],
                stdout=self.tmp, stderr=subprocess.DEVNULL)
            time.sleep(0.3)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        time.sleep(0.1)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.tmp.flush()
        self.tmp.seek(0)
        rows = [r.strip().split(",") for r in self.tmp.read().splitlines() if r.strip()]
        os.unlink(self.tmp.name)
        sm, mx, reasons = [], [], set()
        for r in rows:
            if len(r) < 9:
                continue
            try:
                sm.append(float(r[1]))
                mx.append(float(r[2]))
            except ValueError:
                continue
            for name, v in zip(self.NAMES, r[5:9]):
                if v.strip().lower() == "active":
                    reasons.add(name)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "samples": len(sm),
                "reasons": sorted(reasons)}


# ----------------------------------------------------------------------------- workload
def make_pool(n_frames: int, first: int):
    from paper_2602_01035_gb300 import scenes as S
    cache = {}
    frames = []
    rig = None
    for k in range(n_frames):
        rig, _, fr = S.config3(frame=first + k, cache=cache)
        frames.append(fr)
    return rig, frames


# The method's own arithmetic per gated point, counted as in the scope of the path: about
# 10 FP32 operations for back-projection and gate, 30 per neighbour view for transform,
# projection, pixel choice and residual (Eq. 4-6), and 10 for the weight and the cell key;
# the exact (fixed-point or double-float) evaluation the 1e-5 weight tolerance needs costs
# more than this and is not counted.  The peak is one operation per FP32 lane per clock.
METHOD_OPS_BASE = 20
METHOD_OPS_PER_VIEW = 30
FP32_LANES_PER_SM = 128


def hbm_bytes(stage: str, px: int, cells: float, depth_bytes: int):
    """Algorithmic bytes of one launch of an HBM-bound stage (inputs read once, outputs
    written once); None for stages without such a model."""
    if stage == "count":
        return depth_bytes * px + 4 * px            # depth + confidence
    if stage == "emit":
        return CELL_OUT_BYTES * cells
    return None


def fp32_peak_tops(sm_mhz: float, sms: int) -> float:
    return sms * FP32_LANES_PER_SM * sm_mhz * 1e6 / 1e12


def traffic_table():
    """DRAM bytes per launch per kernel from the committed ncu summary, valid only while the
    kernel sources hash to the value recorded beside the counters."""
    import hashlib
    path = os.path.join(ROOT, "profiles", "dram_traffic.txt")
    src = os.path.join(ROOT, "paper_2602_01035_gb300", "csrc")
    h = hashlib.sha1()
    for name in ("ff_kernels.cu", "ff_device.cuh"):
        with open(os.path.join(src, name), "rb") as f:
            h.update(f.read())
    try:
        rows, recorded = {}, None
        with open(path) as f:
            for line in f:
                parts = line.split()
                if not parts or parts[0].startswith("#"):
                    if len(parts) >= 3 and parts[1] == "sources_sha1":
                        recorded = parts[2]
                    continue
                rows[parts[0]] = float(parts[1])
        return rows if recorded == h.hexdigest() else {}
    except OSError:
        return {}


# ----------------------------------------------------------------------------- ranks
def max_over_ranks(ms: float, world: int, device=None) -> float:
    """Duration of the slowest rank's timed region (the job ends with it)."""
    if world == 1:
        return ms
    import torch
    import torch.distributed as dist
    t = torch.tensor([ms], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_rate(units_per_rank: float, world: int, ms: float) -> float:
    """Whole-job throughput: units processed by all ranks over the slowest rank's time."""
    return units_per_rank * world / (ms / 1e3)


# ----------------------------------------------------------------------------- our arm
def run_ours(args, rank, world, local_rank):
    import torch
    from paper_2602_01035_gb300 import fuseflow as F

    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)
    rig, pool = make_pool(args.pool, first=rank * args.pool)
    px = rig.n_pixels
    frame_bytes = pool[0].input_bytes()
    dtensors = []
    for fr in pool:
        d = [torch.from_numpy(x).to(dev) for x in fr.depth]
        c = [torch.from_numpy(x).to(dev) for x in fr.conf]
        r = [torch.from_numpy(x).to(dev) for x in fr.rgb]
        dtensors.append((d, c, r, [t.data_ptr() for t in d], [t.data_ptr() for t in c],
                         [t.data_ptr() for t in r]))
    ff = F.FuseFlow(rig)
    stream = torch.cuda.current_stream(dev)
    sh = stream.cuda_stream
    FPS = args.frames_per_step

    # launch geometry: the autotuner's choice on the pool's first frame (untimed set-up);
    # every context of this rig takes the same setting (the tile height moves fused values
    # in their last bits only, and a batch needs one tile height)
    tuning = {"autotuned": False, "chosen": ff.tuning()}
    if not args.no_autotune:
        d0 = dtensors[0]
        tu, us0, us1 = ff.autotune(d0[0], d0[1], d0[2], reps=9, stream=sh)
        tuning = {"autotuned": True, "chosen": tu.as_dict(), "start_frame_us": round(us0, 2),
                  "chosen_frame_us": round(us1, 2),
                  "method": "fuseflow_autotune: coordinate descent, median of 9 L2-flushed "
                            "frames per candidate, kept when >= 1% faster"}

    def tuned(ctx_obj):
        g = tuning["chosen"]
        ctx_obj.set_tuning(g["count_chunks"], g["emit_blocks"], g["prefetch_tiles"], g["programmatic"],
                           g["tile_h"])
        return ctx_obj

    def step():
        for i in range(FPS):
            t = dtensors[i % len(dtensors)]
            F.fuseflow_fuse_frame(ff.ctx, t[3], t[4], t[5], sh)

    for _ in range(max(args.warmup, 1)):
        step()
    status, st = ff.stats(sh, check=False)
    if status != F.FUSEFLOW_OK:
        raise RuntimeError(f"fusion failed during warm-up: {F.fuseflow_status_string(status)}")
    n_cells = st.n_cells

    # ------------------------------------------------------------ plain path (one frame per call)
    if world > 1:
        torch.distributed.barrier()
    torch.cuda.synchronize(dev)
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(args.steps):
        step()
    e1.record(stream)
    torch.cuda.synchronize(dev)
    if world > 1:
        torch.distributed.barrier()
    ms = max_over_ranks(e0.elapsed_time(e1), world, dev)
    status, st = ff.stats(sh, check=False)
    ok_status = status == F.FUSEFLOW_OK

    value = job_rate(args.steps * FPS * px, world, ms)
    fps = job_rate(args.steps * FPS, world, ms)

    # ------------------------------------------------------------ recorded fuse calls
    # one CUDA graph per pool frame (fuseflow_graph_*: the five kernels of a frame
    # in one launch), replayed in the plain path's order on the same stream
    graphs = [ff.graph(t[0], t[1], t[2]) for t in dtensors]

    def graph_step():
        for i in range(FPS):
            F.fuseflow_graph_launch(graphs[i % len(graphs)].g, sh)

    for _ in range(max(args.warmup, 1)):
        graph_step()
    g0, g1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    if world > 1:
        torch.distributed.barrier()
    g0.record(stream)
    for _ in range(args.steps):
        graph_step()
    g1.record(stream)
    torch.cuda.synchronize(dev)
    gms = max_over_ranks(g0.elapsed_time(g1), world, dev)
    gstatus, _ = ff.stats(sh, check=False)
    for g in graphs:
        g.close()
    graph_line = {"value": round(job_rate(args.steps * FPS * px, world, gms), 1), "unit": "px/s",
                  "frames_per_s": round(job_rate(args.steps * FPS, world, gms), 2),
                  "ms_per_step": round(gms / args.steps, 4), "vs_plain": round(ms / gms, 4),
                  "status_ok": gstatus == F.FUSEFLOW_OK,
                  "path": "fuseflow_graph_launch, one recorded graph per pool frame"}

    # ------------------------------------------------------------ batched: frames in flight
    # the same frames through `slots` contexts on as many streams, frame k on slot k % slots
    batched = None
    if args.slots > 1:
        B = args.slots
        # several frames in flight: plain stream order (the streams fill the kernel
        # boundaries; levels 0, 1 and 2 measure within 1 % of each other here)
        ctxs = [ff] + [tuned(F.FuseFlow(rig)) for _ in range(B - 1)]
        g_ = tuning["chosen"]
        for c_ in ctxs:
            c_.set_tuning(g_["count_chunks"], g_["emit_blocks"], g_["prefetch_tiles"], 0, g_["tile_h"])
        streams = [stream] + [torch.cuda.Stream(dev) for _ in range(B - 1)]

        def batched_step():
            for i in range(FPS):
                t = dtensors[i % len(dtensors)]
                F.fuseflow_fuse_frame(ctxs[i % B].ctx, t[3], t[4], t[5], streams[i % B].cuda_stream)

        def run_batched(n_steps):
            start = torch.cuda.Event(enable_timing=True)
            stop = torch.cuda.Event(enable_timing=True)
            start.record(stream)
            for s_ in streams[1:]:
                s_.wait_event(start)
            for _ in range(n_steps):
                batched_step()
            for s_ in streams[1:]:
                ev = torch.cuda.Event()
                ev.record(s_)
                stream.wait_event(ev)
            stop.record(stream)
            torch.cuda.synchronize(dev)
            return start.elapsed_time(stop)

        run_batched(max(args.warmup, 1))
        if world > 1:
            torch.distributed.barrier()
        bms = max_over_ranks(run_batched(args.steps), world, dev)
        bst = [c.stats(stream.cuda_stream if k == 0 else streams[k].cuda_stream, check=False)[0]
               for k, c in enumerate(ctxs)]
        batched = {"slots": B, "value": round(job_rate(args.steps * FPS * px, world, bms), 1),
                   "unit": "px/s", "frames_per_s": round(job_rate(args.steps * FPS, world, bms), 2),
                   "ms_per_step": round(bms / args.steps, 4),
                   "vs_plain": round(ms / bms, 4),
                   "status_ok": all(x == F.FUSEFLOW_OK for x in bst),
                   "path": f"{B} contexts on {B} streams, frame k on slot k mod {B}; same frames, "
                           f"CUDA events around the step"}
        for c in ctxs[1:]:
            c.close()
        tuned(ff)                               # the chosen setting again for the lines below

    # ------------------------------------------------------------ batched launch
    # 4 frames per launch sequence (fuseflow_batch: every frame kernel launched once for the
    # 4 frames, 4 contexts), replayed from recorded batch graphs over the pool's frames;
    # per-batch latency from CUDA events on the stream
    # (the headline: the timed region, clocks sampled during it)
    clk = ClockSampler(local_rank)
    batched_launch = run_batched_launch(F, torch, dev, stream, rig, dtensors, tuning, FPS,
                                        args.steps, args.warmup, ms, world, clock=clk)
    clocks = batched_launch.pop("clocks")
    two = run_batched_launch(F, torch, dev, stream, rig, dtensors, tuning, FPS, args.steps, args.warmup,
                             ms, world, n_streams=2)
    two.pop("clocks")
    batched_launch["two_streams"] = two

    # ------------------------------------------------------------ Sec. II.5(2)a top-3 variant
    # (consistency and weights for each cell's 3 most confident members only): same frames,
    # plain path, CUDA events around the step
    top3 = None
    if True:
        ff3 = F.FuseFlow(rig, top_k=3)
        if not args.no_autotune:
            d0 = dtensors[0]
            tu3, _, _ = ff3.autotune(d0[0], d0[1], d0[2], reps=9, stream=sh)
            tuning["chosen_top3"] = tu3.as_dict()

        def top3_step():
            for i in range(FPS):
                t = dtensors[i % len(dtensors)]
                F.fuseflow_fuse_frame(ff3.ctx, t[3], t[4], t[5], sh)

        for _ in range(max(args.warmup, 1)):
            top3_step()
        a0, a1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        if world > 1:
            torch.distributed.barrier()
        a0.record(stream)
        for _ in range(args.steps):
            top3_step()
        a1.record(stream)
        torch.cuda.synchronize(dev)
        tms = max_over_ranks(a0.elapsed_time(a1), world, dev)
        s3, st3 = ff3.stats(sh, check=False)
        F.fuseflow_enable_stage_timing(ff3.ctx, True)
        for i in range(min(FPS, 64)):
            t = dtensors[i % len(dtensors)]
            F.fuseflow_fuse_frame(ff3.ctx, t[3], t[4], t[5], sh)
        st_ms, n_t = F.fuseflow_read_stage_times(ff3.ctx)
        top3 = {"value": round(job_rate(args.steps * FPS * px, world, tms), 1), "unit": "px/s",
                "frames_per_s": round(job_rate(args.steps * FPS, world, tms), 2),
                "ms_per_step": round(tms / args.steps, 4), "vs_plain": round(ms / tms, 4),
                "status_ok": s3 == F.FUSEFLOW_OK, "cells_per_frame": int(st3.n_cells),
                "stage_ms": {k: round(v / max(n_t, 1), 5) for k, v in st_ms.items()},
                "path": "top_k = 3: each cell fuses its 3 most confident members, whose "
                        "consistency is computed per cell in the reduce step"}
        ff3.close()

    # ------------------------------------------------------------ per-frame latency (plain path)
    lat = []
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
           for _ in range(min(FPS, 300))]
    for i, (a, b) in enumerate(evs):
        t = dtensors[i % len(dtensors)]
        a.record(stream)
        F.fuseflow_fuse_frame(ff.ctx, t[3], t[4], t[5], sh)
        b.record(stream)
    torch.cuda.synchronize(dev)
    lat = sorted(a.elapsed_time(b) for a, b in evs)
    p50 = lat[len(lat) // 2]
    p99 = lat[min(len(lat) - 1, int(round(0.99 * (len(lat) - 1))))]

    # ------------------------------------------------------------ per-stage times (roofline)
    F.fuseflow_enable_stage_timing(ff.ctx, True)
    n_stage_frames = min(FPS, 256)
    for i in range(n_stage_frames):
        t = dtensors[i % len(dtensors)]
        F.fuseflow_fuse_frame(ff.ctx, t[3], t[4], t[5], sh)
    stage_ms, n_timed = F.fuseflow_read_stage_times(ff.ctx)
    F.fuseflow_enable_stage_timing(ff.ctx, False)
    stage_avg = {k: v / max(n_timed, 1) for k, v in stage_ms.items()}
    dominant = max(stage_avg, key=stage_avg.get)
    peak, peak_kind = load_peaks()
    depth_bytes = 2
    sm_mhz = float(clocks.get("sm_max_mhz") or 2070.0) if clocks else 2070.0
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    traffic = traffic_table()
    k1 = min(4, rig.n_cams) - 1
    stages = {}
    path_bytes = 9 * px + CELL_OUT_BYTES * n_cells
    for name, t_ms in stage_avg.items():
        alg = hbm_bytes(name, px, n_cells, depth_bytes)
        if name == "assign":
            # the path's algorithmic bytes (inputs read once, the cloud written once) over
            # this kernel's live time, against the measured HBM copy bandwidth; the FP32
            # view beside it counts the method's own operations only
            ach = path_bytes / (t_ms / 1e3) / 1e9
            ops = st.n_gated * (METHOD_OPS_BASE + METHOD_OPS_PER_VIEW * k1)
            fpk = fp32_peak_tops(sm_mhz, sms)
            ach_ops = ops / (t_ms / 1e3) / 1e12
            stages[name] = {"bound": "hbm", "achieved": round(ach, 1), "peak": peak, "unit": "GB/s",
                            "frac": round(ach / peak, 4), "traffic": traffic.get(name),
                            "launch_ms": round(t_ms, 5), "algorithmic_bytes_per_launch": int(path_bytes),
                            "bytes_model": "9 B per input pixel (uint16 depth, float32 confidence, "
                                           "8-bit RGB) + 44 B per output cell",
                            "peak_source": peak_kind,
                            "fp32_view": {"achieved": round(ach_ops, 3), "peak": round(fpk, 2),
                                          "unit": "T op/s", "frac": round(ach_ops / fpk, 4),
                                          "ops_per_launch": int(ops),
                                          "ops_model": f"{METHOD_OPS_BASE} + {METHOD_OPS_PER_VIEW} "
                                                       "(K-1) per gated point, method arithmetic "
                                                       "only (no exact-evaluation overhead)",
                                          "peak_source": f"{sms} SMs x {FP32_LANES_PER_SM} FP32 "
                                                         f"lanes x {sm_mhz:.0f} MHz"}}
        elif alg is not None:
            ach = alg / (t_ms / 1e3) / 1e9
            stages[name] = {"bound": "hbm", "achieved": round(ach, 1), "peak": peak, "unit": "GB/s",
                            "frac": round(ach / peak, 4), "traffic": traffic.get(name),
                            "launch_ms": round(t_ms, 5), "algorithmic_bytes_per_launch": int(alg),
                            "peak_source": peak_kind}
    roof = dict(stages[dominant], kernel=dominant) if dominant in stages else None
    frame_ms = sum(stage_avg.values())
    path_roof = {"bytes_per_frame": int(path_bytes), "frame_ms_staged": round(frame_ms, 5),
                 "achieved_gbs": round(path_bytes / (ms / 1e3 / (args.steps * FPS)) / 1e9, 1),
                 "frac": round(path_bytes / (ms / 1e3 / (args.steps * FPS)) / 1e9 / peak, 4)}

    # ------------------------------------------------------------ Eq. 3 confidence producer
    # (an optional input stage: callers without a confidence image), timed alone over the
    # pool's depth maps (inputs larger than L2), CUDA events on the launching stream
    conf_out = [torch.empty(x.shape, dtype=torch.float32, device=dev) for x in pool[0].depth]
    conf_ptrs = [t.data_ptr() for t in conf_out]
    for i in range(3):
        F.fuseflow_confidence(ff.ctx, dtensors[i % len(dtensors)][3], conf_ptrs, sh)
    c0, c1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    n_conf = 200
    c0.record(stream)
    for i in range(n_conf):
        F.fuseflow_confidence(ff.ctx, dtensors[i % len(dtensors)][3], conf_ptrs, sh)
    c1.record(stream)
    torch.cuda.synchronize(dev)
    conf_ms = c0.elapsed_time(c1) / n_conf
    conf_bytes = (depth_bytes + 4) * px
    stages["confidence"] = {"bound": "hbm", "achieved": round(conf_bytes / (conf_ms / 1e3) / 1e9, 1),
                            "peak": peak, "unit": "GB/s",
                            "frac": round(conf_bytes / (conf_ms / 1e3) / 1e9 / peak, 4),
                            "traffic": traffic.get("confidence"), "launch_ms": round(conf_ms, 5),
                            "algorithmic_bytes_per_launch": int(conf_bytes), "peak_source": peak_kind,
                            "note": "optional producer of Eq. 3, not part of the fused step"}

    # ------------------------------------------------------------ depth screen D^r (Eq. 8)
    # (an optional stage, off by default): the screen alone over the pool's depth maps, and
    # whole frames fused with the edge and range screen set, CUDA events on the stream
    ffs = F.FuseFlow(rig, screen_edge_rel=0.05, screen_min_m=0.3, screen_max_m=8.0)
    scr_out = [torch.empty_like(t) for t in dtensors[0][0]]
    scr_ptrs = [t.data_ptr() for t in scr_out]
    for i in range(3):
        F.fuseflow_screen_depth(ffs.ctx, dtensors[i % len(dtensors)][3], scr_ptrs, sh)
    s0, s1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    n_scr = 200
    s0.record(stream)
    for i in range(n_scr):
        F.fuseflow_screen_depth(ffs.ctx, dtensors[i % len(dtensors)][3], scr_ptrs, sh)
    s1.record(stream)
    torch.cuda.synchronize(dev)
    scr_ms = s0.elapsed_time(s1) / n_scr
    scr_bytes = 2 * depth_bytes * px
    stages["screen"] = {"bound": "hbm", "achieved": round(scr_bytes / (scr_ms / 1e3) / 1e9, 1),
                        "peak": peak, "unit": "GB/s",
                        "frac": round(scr_bytes / (scr_ms / 1e3) / 1e9 / peak, 4),
                        "traffic": traffic.get("screen"), "launch_ms": round(scr_ms, 5),
                        "algorithmic_bytes_per_launch": int(scr_bytes), "peak_source": peak_kind,
                        "note": "optional D^r of Eq. 8 (edge and range screen), off by default"}
    if not args.no_autotune:
        d0 = dtensors[0]
        ffs.autotune(d0[0], d0[1], d0[2], reps=9, stream=sh)
    for i in range(4):
        t = dtensors[i % len(dtensors)]
        F.fuseflow_fuse_frame(ffs.ctx, t[3], t[4], t[5], sh)
    n_sf = min(FPS, 200)
    s0.record(stream)
    for i in range(n_sf):
        t = dtensors[i % len(dtensors)]
        F.fuseflow_fuse_frame(ffs.ctx, t[3], t[4], t[5], sh)
    s1.record(stream)
    torch.cuda.synchronize(dev)
    sfs_ms = s0.elapsed_time(s1) / n_sf
    sst, sstats = ffs.stats(sh, check=False)
    screened = {"frames_per_s": round(1e3 / sfs_ms, 2), "vs_plain": round((ms / (args.steps * FPS)) / sfs_ms, 4),
                "status_ok": sst == F.FUSEFLOW_OK, "n_valid": int(sstats.n_valid),
                "n_valid_unscreened": int(st.n_valid), "cells_per_frame": int(sstats.n_cells),
                "settings": "screen_edge_rel 0.05, screen_min_m 0.3, screen_max_m 8.0"}
    ffs.close()

    # ------------------------------------------------------------ end to end (host buffers)
    # The public serving API on this rig: frames from pinned host memory, results into
    # pinned host arrays, `slots` frames in flight (copies overlap other frames' kernels).
    from collections import deque
    from paper_2602_01035_gb300 import serving as SV
    n_e2e = max(1, min(args.e2e_frames, FPS))
    B = max(1, args.slots)
    pinned = [SV.pinned_frame(fr) for fr in pool]
    cap = ff.capacity
    srv = SV.Server(1 << 40)
    rid = srv.add_rig(rig, n_slots=B)
    srv.reserve(rid, B)
    if not args.no_autotune:
        srv.autotune(rid, pinned[0], reps=9)
    outs = deque(SV.HostCloud(cap) for _ in range(B + 1))

    def serve(n_frames):
        sent, got, d2h_bytes, flying = 0, 0, 0, {}
        while got < n_frames:
            while sent < n_frames and outs:
                buf = outs.popleft()
                flying[srv.submit(rid, pinned[sent % len(pinned)], buf)] = buf
                sent += 1
            for req, _, status, st_ in srv.poll():
                outs.append(flying.pop(req))
                d2h_bytes += st_["n_cells"] * CELL_OUT_BYTES + 48
                got += 1
        return d2h_bytes

    serve(2 * B)
    if world > 1:
        torch.distributed.barrier()
    t0 = time.perf_counter()
    d2h = serve(n_e2e)
    e2e_s = max_over_ranks((time.perf_counter() - t0) * 1e3, world, dev) / 1e3
    srv.close()
    e2e = {"value": round(job_rate(n_e2e * px, world, e2e_s * 1e3), 1), "unit": "px/s",
           "frames_per_s": round(job_rate(n_e2e, world, e2e_s * 1e3), 2),
           "h2d_bytes_per_step": int(frame_bytes * FPS),
           "d2h_bytes_per_step": int(d2h / n_e2e * FPS),
           "frames_timed": n_e2e, "slots": B,
           "entry_point": "fuseflow_server_submit / fuseflow_server_poll (host buffers)"}
    # the synchronous single-call host entry point, for reference
    ctx_host = [SV.HostCloud(cap)]
    h = ctx_host[0].c
    fr0 = pinned[0]                               # untimed: the staging buffers' first use
    F.fuseflow_fuse_frame_host(ff.ctx, fr0["depth"], fr0["conf"], fr0["rgb"], h.pos, h.rgb,
                               h.weight, h.count, h.rep, h.key, sh)
    t0 = time.perf_counter()
    n_single = min(64, n_e2e)
    for i in range(n_single):
        fr = pinned[i % len(pinned)]
        F.fuseflow_fuse_frame_host(ff.ctx, fr["depth"], fr["conf"], fr["rgb"], h.pos, h.rgb,
                                   h.weight, h.count, h.rep, h.key, sh)
    e2e["single_call_frames_per_s"] = round(n_single / (time.perf_counter() - t0), 2)

    # ------------------------------------------------------------ the other configurations
    configs, groups = None, {}
    if rank == 0 and world == 1 and not args.no_serving:
        configs, groups = run_configs(dev)

    # ------------------------------------------------------------ served vs plain
    # in a fresh process on the same GPU (this one stays idle meanwhile): the latency tail of
    # a wall-clock replay measured inside this long-running process came out 15-30 times
    # longer, for the served and the plain path alike, than in a process of its own
    serving = None
    if rank == 0 and world == 1 and not args.no_serving:
        import multiprocessing as mp
        import queue as _queue
        torch.cuda.synchronize(dev)
        ctx_ = mp.get_context("spawn")
        q_ = ctx_.Queue()
        child = ctx_.Process(target=serving_child, args=(vars(args), local_rank, q_))
        child.start()                    # not a pool worker: it renders with a pool itself
        try:
            serving = q_.get(timeout=3600)
        except _queue.Empty:
            serving = {"error": "the serving replay process returned nothing"}
        child.join()

    # ------------------------------------------------------------ CPU baseline (oracle)
    cpu, parity = None, None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cpu = cpu_baseline(rig, pool[:8])
        cpu["all_cores"] = cpu_baseline_all_cores(rig, pool[:8])
        cases = [("cfg3_8x1280x720", rig, pool[0])]
        for key, label in (("cfg1", "cfg1_2x160x120"), ("cfg2", "cfg2_4x640x480"),
                           ("cfg4_2cams", "cfg4_2x1024x1024"), ("cfg4_8cams", "cfg4_8x1024x1024"),
                           ("cfg4_16cams", "cfg4_16x1024x1024"), ("cfg4_32cams", "cfg4_32x1024x1024")):
            if key in groups:
                cases.append((label, groups[key][0], groups[key][1][0]))
        parity = parity_block(dev, cases)

    bl = batched_launch
    out = {
        "metric": METRIC, "value": bl["value"], "unit": "px/s", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": bl["ms_per_step"], "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": "8x1280x720 rig: uint16 depth (mm), float32 confidence, uint8 RGB; "
                               f"{FPS} frames per step, {bl['frames_per_batch']} frames per batched "
                               "launch (every frame kernel launched once for them) replayed from "
                               "captured CUDA graphs",
                   "n_cams": 8, "width": 1280, "height": 720, "frames_per_step": FPS,
                   "pool_frames": len(pool), "pool_bytes": int(frame_bytes * len(pool)),
                   "l2": "inputs larger than L2: a pool of distinct frames is cycled, each frame "
                         "re-read only after the others",
                   "parallelism": f"replicas x{world}", "launch_geometry": tuning},
        "frames_per_s": bl["frames_per_s"],
        "latency_ms": dict(bl["latency_ms"]),
        "plain_path": {"value": round(value, 1), "unit": "px/s", "frames_per_s": round(fps, 2),
                       "ms_per_step": round(ms / args.steps, 4),
                       "latency_ms": {"p50": round(p50, 5), "p99": round(p99, 5)},
                       "path": "one frame per fuseflow_fuse_frame call, one stream"},
        "roofline": roof, "path_roofline": path_roof,
        "stage_ms": {k: round(v, 5) for k, v in stage_avg.items()},
        "stage_roofline": stages,
        "graph_replay": graph_line, "batched": batched, "batched_launch": batched_launch,
        "top3_variant": top3,
        "screened_variant": screened, "serving": serving, "other_configs": configs,
        "e2e": e2e, "gpu_launches": int(bl["kernel_launches"]),
        "cells_per_frame": int(n_cells), "status_ok": ok_status,
        "clocks": clocks, "cpu_baseline": cpu, "parity": parity,
    }
    ff.close()
    if world > 1:
        torch.distributed.destroy_process_group()
    if rank == 0:
        print(json.dumps(out), flush=True)


# ----------------------------------------------------------------------------- batched launch
def run_batched_launch(F, torch, dev, stream, rig, dtensors, tuning, FPS, steps, warmup, ms_plain,
                       world, B=4, n_streams=1, clock=None):
    """Frames of the benchmark rig fused B at a time by one launch of each frame kernel
    (fuseflow_batch), each batch replayed from a recorded graph over fixed pool frames;
    with n_streams > 1, consecutive batches alternate over that many streams (one batch
    object of B contexts each), so one batch's kernels overlap the next one's."""
    g_ = tuning["chosen"]
    pdl = g_["programmatic"] if n_streams == 1 else 0
    ctxs = [F.FuseFlow(rig) for _ in range(B * n_streams)]
    for c in ctxs:
        c.set_tuning(g_["count_chunks"], g_["emit_blocks"], g_["prefetch_tiles"], pdl, g_["tile_h"])
    batches = [F.Batch(ctxs[k * B:(k + 1) * B]) for k in range(n_streams)]
    streams = [stream] + [torch.cuda.Stream(dev) for _ in range(n_streams - 1)]
    n_groups = max(1, len(dtensors) // B)
    groups = [[dtensors[(k * B + i) % len(dtensors)][:3] for i in range(B)] for k in range(n_groups)]
    graphs = [[b.graph(gr) for gr in groups] for b in batches]
    n_batches = FPS // B

    def step():
        for k in range(n_batches):
            q = k % n_streams
            F.fuseflow_graph_launch(graphs[q][(k // n_streams) % n_groups].g, streams[q].cuda_stream)

    def run(n_steps):
        a = torch.cuda.Event(enable_timing=True)
        b = torch.cuda.Event(enable_timing=True)
        a.record(stream)
        for s_ in streams[1:]:
            s_.wait_event(a)
        for _ in range(n_steps):
            step()
        for s_ in streams[1:]:
            ev = torch.cuda.Event()
            ev.record(s_)
            stream.wait_event(ev)
        b.record(stream)
        torch.cuda.synchronize(dev)
        return a.elapsed_time(b)

    run(max(warmup, 1))
    if clock is not None:
        clock.start()
    if world > 1:
        torch.distributed.barrier()
    bms = run(steps)
    if world > 1:
        torch.distributed.barrier()
    clocks = clock.stop() if clock is not None else None
    bms = max_over_ranks(bms, world, dev)
    frames = steps * n_batches * B
    # per-batch latency on one stream, back to back (each of its B frames completes with it)
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(200)]
    for k, (a, b) in enumerate(evs):
        a.record(stream)
        F.fuseflow_graph_launch(graphs[0][k % n_groups].g, stream.cuda_stream)
        b.record(stream)
    torch.cuda.synchronize(dev)
    lat = sorted(a.elapsed_time(b) for a, b in evs)
    ok = all(c.stats(stream.cuda_stream, check=False)[0] == F.FUSEFLOW_OK for c in ctxs)
    for gs in graphs:
        for g in gs:
            g.close()
    for b in batches:
        b.close()
    for c in ctxs:
        c.close()
    px = rig.n_pixels
    plain_fps = steps * FPS / (ms_plain / 1e3)
    return {"frames_per_batch": B, "streams": n_streams,
            "value": round(job_rate(frames * px, world, bms), 1), "unit": "px/s",
            "frames_per_s": round(job_rate(frames, world, bms), 2),
            "ms_per_step": round(bms / steps, 4),
            "vs_plain": round(job_rate(frames, world, bms) / (plain_fps * world), 4),
            "latency_ms": {"p50": round(lat[len(lat) // 2], 5),
                           "p99": round(lat[min(len(lat) - 1, int(round(0.99 * (len(lat) - 1))))], 5),
                           "of": "one batch of B frames alone on a stream (its B frames complete with it)"},
            "status_ok": ok, "clocks": clocks, "kernel_launches": steps * n_batches * KERNELS_PER_FRAME,
            "path": f"fuseflow_batch over {B} contexts: each frame kernel launched once for the {B} "
                    f"frames, recorded as graphs over groups of pool frames, replayed on {n_streams} "
                    "stream(s)"}


def run_mixed_batch(F, torch, dev, groups, reps=64):
    """One frame each of several rigs (the 2/8/16/32-camera 1024x1024 sweep) fused by one
    batched launch (replayed graph) against the same frames fused one call after another."""
    stream = torch.cuda.current_stream(dev)
    sh = stream.cuda_stream
    rigs = [groups[k][0] for k in groups]
    frs = [groups[k][1][0] for k in groups]
    dev_frames = []
    for fr in frs:
        d = [torch.from_numpy(x).to(dev) for x in fr.depth]
        c = [torch.from_numpy(x).to(dev) for x in fr.conf]
        r = [torch.from_numpy(x).to(dev) for x in fr.rgb]
        dev_frames.append((d, c, r))
    ctxs = [F.FuseFlow(rig) for rig in rigs]
    for c, t in zip(ctxs, dev_frames):
        c.autotune(t[0], t[1], t[2], reps=9, stream=sh)
    # one assign kernel serves the batch: every context takes the tile height chosen for the
    # rig with the most pixels
    th = ctxs[max(range(len(ctxs)), key=lambda i: ctxs[i].n_pixels)].tuning()["tile_h"]
    for c in ctxs:
        tu_ = c.tuning()
        c.set_tuning(tu_["count_chunks"], tu_["emit_blocks"], tu_["prefetch_tiles"], tu_["programmatic"], th)
    batch = F.Batch(ctxs)
    g = batch.graph(dev_frames)
    plain = [c.graph(*t) for c, t in zip(ctxs, dev_frames)]
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)

    def timed(fn):
        for _ in range(3):
            fn()
        e0.record(stream)
        for _ in range(reps):
            fn()
        e1.record(stream)
        torch.cuda.synchronize(dev)
        return e0.elapsed_time(e1) / reps

    t_batch = timed(lambda: F.fuseflow_graph_launch(g.g, sh))
    t_plain = timed(lambda: [F.fuseflow_graph_launch(p.g, sh) for p in plain])
    ok = all(c.stats(sh, check=False)[0] == F.FUSEFLOW_OK for c in ctxs)
    px = sum(r.n_pixels for r in rigs)
    g.close()
    for p in plain:
        p.close()
    batch.close()
    for c in ctxs:
        c.close()
    return {"rigs": [f"{r.n_cams}x{r.cameras[0].width}x{r.cameras[0].height}" for r in rigs],
            "batch_ms": round(t_batch, 4), "plain_ms": round(t_plain, 4),
            "px_per_s_batch": round(px / (t_batch / 1e3), 1), "px_per_s_plain": round(px / (t_plain / 1e3), 1),
            "vs_plain": round(t_plain / t_batch, 4), "status_ok": ok,
            "path": "one batched launch (recorded graph) vs the four recorded plain calls in a row"}


# ----------------------------------------------------------------------------- other configs
def run_configs(dev, frames_each: int = 64):
    """Device-resident throughput of the other rigs on the plain path (one frame per fuse
    call, CUDA events on the launching stream): 2x160x120 float32, 4x640x480, and the
    2/8/16/32-camera 1024x1024 rig-scaling sweep."""
    import multiprocessing as mp
    import torch
    from paper_2602_01035_gb300 import fuseflow as F
    from paper_2602_01035_gb300 import scenes as S

    specs = [("cfg1",), ("cfg2", 0), ("cfg2", 1), ("cfg4", 2), ("cfg4", 8), ("cfg4", 16), ("cfg4", 32)]
    with mp.get_context("spawn").Pool(min(len(specs), os.cpu_count() or 1)) as pool:
        rendered = pool.map(S.config_frame, specs)
    groups = {}
    for spec, (rig, fr) in zip(specs, rendered):
        key = spec[0] if spec[0] != "cfg4" else f"cfg4_{spec[1]}cams"
        groups.setdefault(key, (rig, []))[1].append(fr)
    stream = torch.cuda.current_stream(dev)
    out = {}
    if "cfg2" in groups:
        out["table2_shape"] = run_ablations(dev, *groups["cfg2"])
    out["cfg4_mixed_batch"] = run_mixed_batch(F, torch, dev, {k: v for k, v in groups.items()
                                                             if k.startswith("cfg4_")})
    for key, (rig, frs) in groups.items():
        dev_frames = []
        for fr in frs:
            d = [torch.from_numpy(x).to(dev) for x in fr.depth]
            c = [torch.from_numpy(x).to(dev) for x in fr.conf]
            r = [torch.from_numpy(x).to(dev) for x in fr.rgb]
            dev_frames.append((d, c, r, [t.data_ptr() for t in d], [t.data_ptr() for t in c],
                               [t.data_ptr() for t in r]))
        ff = F.FuseFlow(rig)
        t0_ = dev_frames[0]
        tu, us0, us1 = ff.autotune(t0_[0], t0_[1], t0_[2], reps=9, stream=stream.cuda_stream)
        for i in range(4):
            t = dev_frames[i % len(dev_frames)]
            F.fuseflow_fuse_frame(ff.ctx, t[3], t[4], t[5], stream.cuda_stream)
        n_fr = frames_each if rig.n_pixels > (1 << 21) else 4 * frames_each   # small rigs: more
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for i in range(n_fr):
            t = dev_frames[i % len(dev_frames)]
            F.fuseflow_fuse_frame(ff.ctx, t[3], t[4], t[5], stream.cuda_stream)
        e1.record(stream)
        torch.cuda.synchronize(dev)
        ms = e0.elapsed_time(e1)
        status, st = ff.stats(stream.cuda_stream, check=False)
        px = rig.n_pixels
        # the same frames replayed from recorded graphs (one per distinct frame)
        graphs = [ff.graph(t[0], t[1], t[2]) for t in dev_frames]
        for i in range(4):
            F.fuseflow_graph_launch(graphs[i % len(graphs)].g, stream.cuda_stream)
        e0.record(stream)
        for i in range(n_fr):
            F.fuseflow_graph_launch(graphs[i % len(graphs)].g, stream.cuda_stream)
        e1.record(stream)
        torch.cuda.synchronize(dev)
        gms = e0.elapsed_time(e1)
        for g in graphs:
            g.close()
        out[key] = {"cams": rig.n_cams, "px_per_frame": px, "frames_per_s": round(n_fr / (ms / 1e3), 2),
                    "px_per_s": round(n_fr * px / (ms / 1e3), 1),
                    "px_per_s_per_camera": round(n_fr * px / (ms / 1e3) / rig.n_cams, 1),
                    "cells": int(st.n_cells), "status_ok": status == F.FUSEFLOW_OK,
                    "graph_frames_per_s": round(n_fr / (gms / 1e3), 2), "frames_timed": n_fr,
                    "launch_geometry": dict(tu.as_dict(), start_frame_us=round(us0, 2),
                                            chosen_frame_us=round(us1, 2))}
        ff.close()
    return out, groups


def run_ablations(dev, rig, frames, frames_each: int = 64):
    """Table II's comparison on the 4-camera dynamic rig: E_MC (Eq. 12, millimetres, mean
    over the frames) and frames/s of the full method, without measurement confidence
    (no gate, omega = V), without distance consistency (V = 1), and without the spatial
    hash (point-wise: every gated point is an output point; no fusion path is timed)."""
    import numpy as np
    import torch
    from paper_2602_01035_gb300 import fuseflow as F
    stream = torch.cuda.current_stream(dev)
    sh = stream.cuda_stream
    dev_frames = []
    for fr in frames:
        d = [torch.from_numpy(x).to(dev) for x in fr.depth]
        c = [torch.from_numpy(x).to(dev) for x in fr.conf]
        r = [torch.from_numpy(x).to(dev) for x in fr.rgb]
        dev_frames.append((d, c, r, [t.data_ptr() for t in d], [t.data_ptr() for t in c],
                           [t.data_ptr() for t in r]))
    modes = {"full": {}, "full_top3": {"top_k": 3}, "no_MF": {"use_conf": 0},
             "no_DC": {"use_consistency": 0}}
    res = {}
    for name, prm in modes.items():
        ff = F.FuseFlow(rig, **prm)
        mcs = []
        for t in dev_frames:
            cloud = F.fuseflow_fuse_frame(ff.ctx, t[3], t[4], t[5], sh)
            _, st = ff.stats(sh, check=False)
            mc, _ = F.fuseflow_mc_error(ff.ctx, cloud.pos, st.n_cells, t[3], stream=sh)
            mcs.append(mc * 1e3)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for i in range(frames_each):
            t = dev_frames[i % len(dev_frames)]
            F.fuseflow_fuse_frame(ff.ctx, t[3], t[4], t[5], sh)
        e1.record(stream)
        torch.cuda.synchronize(dev)
        res[name] = {"mc_error_mm": round(float(np.mean(mcs)), 3),
                     "frames_per_s": round(frames_each / (e0.elapsed_time(e1) / 1e3), 1)}
        ff.close()
    # point-wise (no spatial hash): every gated pixel an output point with its own weight,
    # consistency over all points (fuseflow_fuse_points), timed like the other modes
    ff = F.FuseFlow(rig)
    npx = rig.n_pixels
    pw = torch.empty((npx, 3), dtype=torch.float32, device=dev)
    wt = torch.empty((npx,), dtype=torch.float32, device=dev)
    col = torch.empty((npx, 3), dtype=torch.uint8, device=dev)
    mcs = []
    for t in dev_frames:
        F.fuseflow_fuse_points(ff.ctx, t[3], t[4], t[5], pw.data_ptr(), wt.data_ptr(), col.data_ptr(), sh)
        pts = pw[torch.isfinite(pw[:, 0])].contiguous()
        mc, _ = F.fuseflow_mc_error(ff.ctx, pts.data_ptr(), pts.shape[0], t[3], stream=sh)
        mcs.append(mc * 1e3)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for i in range(frames_each):
        t = dev_frames[i % len(dev_frames)]
        F.fuseflow_fuse_points(ff.ctx, t[3], t[4], t[5], pw.data_ptr(), wt.data_ptr(), col.data_ptr(), sh,
                               counts=False)
    e1.record(stream)
    torch.cuda.synchronize(dev)
    ff.close()
    res["no_SA"] = {"mc_error_mm": round(float(np.mean(mcs)), 3),
                    "frames_per_s": round(frames_each / (e0.elapsed_time(e1) / 1e3), 1),
                    "path": "fuseflow_fuse_points: point-wise output, consistency for every gated point"}
    res["note"] = (f"{rig.n_cams}x{rig.cameras[0].width}x{rig.cameras[0].height} moving-sphere rig, "
                   f"{len(frames)} frames; E_MC with a {F.MC_OCCLUSION_M} m occlusion margin; full = "
                   "every member fused, full_top3 = each cell's 3 most confident members (the "
                   "paper's order: consistency for those only)")
    return res


# ----------------------------------------------------------------------------- serving
SERVE_BUDGET = 20 << 30          # HBM budget of the served rigs' slots (bytes): binds below
                                 # the 24 slots the 12 rigs ask for


def serving_child(arg_dict, local_rank, out_queue):
    """run_serving in a process of its own (module level, for a spawn context).  The server
    gives each of its slots a stream; with CUDA's default 8 hardware work queues, streams
    that share a queue serialise, which lengthened the latency tail, so this process asks
    for 32 before it initialises CUDA.  The rigs ask for 24 slots in all, under the 32:
    with 36 to 43 slots (3 or 4 per rig) the served p99 of a 30 s trace grew from 5 ms to
    68-140 ms, growing window by window, as frames of different rigs queued behind one
    another in shared queues."""
    os.environ.setdefault("CUDA_DEVICE_MAX_CONNECTIONS", "32")
    import torch
    torch.cuda.set_device(local_rank)
    try:
        res = run_serving(argparse.Namespace(**arg_dict), torch.device("cuda", local_rank))
    except Exception as exc:                     # reported in the JSON line, not raised
        res = {"error": f"{type(exc).__name__}: {exc}"}
    out_queue.put(res)


def run_serving(args, dev):
    """Served vs plain on one seeded Poisson trace over 12 rigs of 2-24 cameras at
    320x240 to 1920x1080 (15-60 fps per rig), frames from pinned host memory."""
    import multiprocessing as mp
    import numpy as np
    import torch
    from paper_2602_01035_gb300 import fuseflow as F
    from paper_2602_01035_gb300 import scenes as S
    from paper_2602_01035_gb300 import serving as SV

    rigs, _ = S.serving_rigs()
    n = len(rigs)
    with mp.get_context("spawn").Pool(min(n, os.cpu_count() or 1)) as pool:
        frames = pool.map(S.serving_frame, range(n))
    rng = np.random.default_rng(5999 + 2)
    rates = rng.uniform(15.0, 60.0, size=n)
    trace = SV.poisson_trace(rates, args.serve_seconds, seed=5999 + 3)
    px = [r.n_pixels for r in rigs]
    pinned = [SV.pinned_frame(f) for f in frames]
    caps = [max(65536, p // 16) for p in px]

    # every rig asks for SERVE_MAX_SLOTS frames in flight, more slots than fit in the budget:
    # they are reserved round-robin until it binds, and frames of rigs below their request
    # wait for memory; the largest rig is removed halfway through the trace (its memory goes
    # to the rigs below their request)
    removals = [(args.serve_seconds / 2.0, int(np.argmax(px)))]

    def served_run(trace_, removals_):
        srv = SV.Server(SERVE_BUDGET)
        rids = [srv.add_rig(rig, n_slots=args.serve_slots, max_cells=caps[r]) for r, rig in enumerate(rigs)]
        held = [1] * n
        for k in range(2, args.serve_slots + 1):         # share the budget evenly, round-robin
            held = [srv.reserve(rid, k) for rid in rids]
        srv.set_max_inflight(args.serve_max_inflight)
        from collections import deque
        outs = [deque(SV.HostCloud(caps[r]) for _ in range(args.serve_slots + 1)) for r in range(n)]
        for r in range(n):                           # warm-up: one frame per rig
            buf = outs[r].popleft()
            srv.submit(rids[r], pinned[r], buf)
            outs[r].append(buf)
        srv.drain()
        before = srv.stats()
        res = SV.replay_served(srv, rids, pinned, outs, trace_, px, removals=removals_)
        after = srv.stats()
        srv.close()
        res["admission"] = {"budget_bytes": SERVE_BUDGET, "slots_asked_per_rig": args.serve_slots,
                            "slots_held_per_rig": held, "hbm_bytes_at_start": int(before["used_bytes"]),
                            "hbm_bytes_at_end": int(after["used_bytes"]),
                            "slots_at_end": int(after["slots"]),
                            **{k: int(after[k] - before[k]) for k in
                               ("deferred_by_budget", "slots_grown", "frames_cancelled", "frames_failed")}}
        return res

    served = served_run(trace, removals)
    sat_trace = [(0.0, r) for _, r in trace]
    served_sat = served_run(sat_trace, [])

    ctxs = [F.FuseFlow(rig, max_cells=caps[r]) for r, rig in enumerate(rigs)]
    plain_outs = [SV.HostCloud(caps[r]) for r in range(n)]
    sh = torch.cuda.current_stream(dev).cuda_stream
    for r in range(n):
        F.fuseflow_fuse_frame_host(ctxs[r].ctx, pinned[r]["depth"], pinned[r]["conf"],
                                   pinned[r]["rgb"], plain_outs[r].c.pos, plain_outs[r].c.rgb,
                                   plain_outs[r].c.weight, plain_outs[r].c.count,
                                   plain_outs[r].c.rep, plain_outs[r].c.key, sh)
    plain = SV.replay_plain([c.ctx for c in ctxs], pinned, plain_outs, trace, px, sh, removals=removals)
    plain_sat = SV.replay_plain([c.ctx for c in ctxs], pinned, plain_outs, sat_trace, px, sh)
    for c in ctxs:
        c.close()
    return {
        "workload": f"{n} rigs of 2-24 cameras, 320x240 to 1920x1080 uint16, Poisson arrivals at "
                    f"15-60 fps per rig for {args.serve_seconds:g} s ({len(trace)} frames, "
                    f"{sum(px) / 1e6:.1f} Mpx per round of all rigs); frames from pinned host memory, "
                    f"results into pinned host arrays; one rendered frame per rig, resubmitted",
        "removal": {"rig": int(removals[0][1]), "at_s": removals[0][0],
                    "rig_shape": f"{rigs[removals[0][1]].n_cams}x{rigs[removals[0][1]].cameras[0].width}"
                                 f"x{rigs[removals[0][1]].cameras[0].height}",
                    "note": "its later arrivals are left out of both replays"},
        "served": dict(served, max_inflight=args.serve_max_inflight),
        "plain": dict(plain, path="one fuseflow_fuse_frame_host call at a time, arrival order"),
        "saturated": {"served_frames_per_s": served_sat["frames_per_s"],
                      "plain_frames_per_s": plain_sat["frames_per_s"],
                      "served_px_per_s": served_sat["px_per_s"], "plain_px_per_s": plain_sat["px_per_s"],
                      "note": "the same frames, all arrived at t = 0"},
    }


# ----------------------------------------------------------------------------- oracle timing
def cpu_baseline(rig, frames, row_step=1):
    from oracle import oracle
    oracle.build()
    t0 = time.perf_counter()
    n = 0
    for fr in frames:
        oracle.fuse_frame(rig, fr, {"row_step": row_step}, points=False)
        n += rig.n_pixels // row_step
    dt = time.perf_counter() - t0
    return {"value": round(n / dt, 1), "unit": "px/s", "cores": 1, "kind": "oracle",
            "sample": f"{len(frames)} frame(s) of the 8x1280x720 rig, rows y % {row_step} == 0 "
                      f"back-projected ({n} px), {dt:.1f} s on one host core"}


def parity_block(dev, cases):
    """Oracle parity of one frame of each configuration (part of the oracle leg): the frame
    is fused on the GPU with its per-pixel cell keys traced, the FP64 oracle fuses it on the
    host (frames in parallel threads: the oracle runs in C without the GIL), and every cell
    outside the oracle's exclusion sets is compared (oracle/compare.py).  Reports the counts
    of compared and excluded cells and of boundary, ambiguous and tie points."""
    import torch
    from concurrent.futures import ThreadPoolExecutor
    from oracle import compare as OC
    from oracle import oracle
    from paper_2602_01035_gb300 import fuseflow as F
    oracle.build()
    gpu = {}
    for label, rig, fr in cases:
        ff = F.FuseFlow(rig)
        d = [torch.from_numpy(x).to(dev) for x in fr.depth]
        c = [torch.from_numpy(x).to(dev) for x in fr.conf]
        r = [torch.from_numpy(x).to(dev) for x in fr.rgb]
        keys = torch.zeros(rig.n_pixels, dtype=torch.int64, device=dev)
        ff.set_trace(key=keys)
        cloud = ff.fuse(d, c, r)
        status, st = ff.stats(check=False)
        ff.clear_trace()
        n = int(st.n_cells)
        cells = {k: v.cpu().numpy().copy() for k, v in ff.cloud_tensors(cloud, n).items()}
        for k, dt in (("count", np.uint32), ("rep", np.uint32), ("key", np.uint64)):
            cells[k] = cells[k].view(dt)
        gpu[label] = ({"status": status, "stats": st.as_dict(), "cells": cells},
                      keys.cpu().numpy().view(np.uint64))
        ff.close()
        del d, c, r, keys

    def one(case):
        label, rig, fr = case
        res, keys = gpu[label]
        try:
            orc = oracle.fuse_frame(rig, fr, {}, cell_capacity=max(1 << 20, rig.n_pixels // 4))
            boundary, amb, tie = OC.point_masks(orc)
            inr = orc["in_range"].astype(bool)
            excl = (boundary | amb) & inr
            rep = OC.compare_cells(res, orc, {}, excl, keys)
            return label, {"pixels": rig.n_pixels, "status_ok": res["status"] == F.FUSEFLOW_OK,
                           "cells_oracle": rep["n_cells_oracle"], "cells_compared": rep["n_cells_matched"],
                           "cells_excluded": rep["n_cells_excluded"],
                           "cells_flagged_by_oracle": rep["n_cells_flagged_by_oracle"],
                           "excluded_fraction": rep["excluded_fraction"],
                           "cells_with_tie_weights": rep["n_tie_cells"],
                           "boundary_points": int((boundary & inr).sum()),
                           "ambiguous_points": int((amb & inr).sum()),
                           "tie_points": int(tie.sum()),
                           "max_w_rel_err": rep["max_w_rel_err"], "max_pos_err_m": rep["max_pos_err_m"],
                           "max_rgb_err": rep["max_rgb_err"], "all_compared_match": True}
        except AssertionError as exc:
            return label, {"pixels": rig.n_pixels, "all_compared_match": False, "failure": str(exc)[:200]}

    t0 = time.perf_counter()
    with ThreadPoolExecutor(max_workers=len(cases)) as ex:
        out = dict(ex.map(one, cases))
    out["note"] = ("frame 0 of each rig; cells outside the oracle's exclusion sets (a member within "
                   "1e-5 m of a cell face, an ambiguous coarse level, and every cell such a point "
                   "reaches on the GPU) compared exactly (count, representative) and within the "
                   "tolerances (W 1e-5 rel, position 1e-5 m + 1e-5 rel, colour 6e-3); tie cells "
                   f"compared structurally only; {time.perf_counter() - t0:.1f} s of oracle work")
    return out


def _oracle_worker(item):
    rig, fr = item
    from oracle import oracle
    oracle.build()
    t0 = time.perf_counter()
    oracle.fuse_frame(rig, fr, {}, points=False)
    return rig.n_pixels, time.perf_counter() - t0


def cpu_baseline_all_cores(rig, frames):
    """The oracle on every host core at once: one process per core, one frame each."""
    import multiprocessing as mp
    n = os.cpu_count() or 1
    items = [(rig, frames[k % len(frames)]) for k in range(n)]
    with mp.get_context("spawn").Pool(n) as pool:
        res = pool.map(_oracle_worker, items)
    px = sum(r[0] for r in res)
    wall = max(r[1] for r in res)
    return {"value": round(px / wall, 1), "unit": "px/s", "cores": n, "kind": "oracle",
            "sample": f"{n} processes, one 8x1280x720 frame each, concurrently; "
                      f"slowest {wall:.1f} s"}


def run_reference(args, rank, world):
    if rank != 0:
        return
    from oracle import oracle
    oracle.build()
    from paper_2602_01035_gb300 import scenes as S
    rig, _, fr = S.config3(frame=0)
    row_step = 8
    px = rig.n_pixels // row_step
    for _ in range(args.warmup):
        oracle.fuse_frame(rig, fr, {"row_step": row_step}, points=False)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        oracle.fuse_frame(rig, fr, {"row_step": row_step}, points=False)
    dt = time.perf_counter() - t0
    value = args.steps * px / dt
    out = {
        "metric": METRIC, "value": round(value, 1), "unit": "px/s", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(dt / args.steps * 1e3, 3),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic", "impl": "reference",
        "config": {"workload": "8x1280x720 rig: uint16 depth (mm), float32 confidence, uint8 RGB; "
                               "each step fuses a row sample of one frame on the host",
                   "n_cams": 8, "width": 1280, "height": 720, "parallelism": "host, 1 core"},
        "cpu_baseline": {"value": round(value, 1), "unit": "px/s", "cores": 1, "kind": "oracle",
                         "sample": f"per step: rows y % {row_step} == 0 of one 8x1280x720 frame "
                                   f"({px} px), all 8 depth maps used by the consistency views"},
        "e2e": {"value": round(value, 1), "unit": "px/s", "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
    }
    print(json.dumps(out), flush=True)


def main():
    args = parse()
    rank, world, local_rank = dist_env()
    if args.impl == "reference":
        run_reference(args, rank, world)
        return
    run_ours(args, rank, world, local_rank)


if __name__ == "__main__":
    main()
