#!/usr/bin/env python
"""ELT-scale SCAO real-time-control benchmark on one GB300 (or N replicas).

One step = one WFS frame through the whole hot path: pixel calibration,
centre-of-gravity slopes and the partial DM vectors of the matrix slices (one
kernel), then their sum and the leaky integrator (a second, overlapping one), on the
74x74-subaperture, 740x740-pixel frame with the 4421 x 7944 control matrix (stored
FP32 by default).

Timing: every step is bracketed by CUDA events on the launching stream, which gives
the frame latency distribution (p50/p99/p99.9, RMS jitter); the two stage calls are
timed the same way, with an event between them.  L2 is flushed between steps by reading a 512 MiB device buffer (a read leaves only
clean lines behind, so no write-back lands inside the next step), outside the
events.  The host
enqueues each batch of steps behind a device-side sleep so that the GPU never
waits on the host inside a timed step.  ``e2e`` repeats the measurement through
the synchronous host-buffer C call (pinned frame in, DM commands out), timed on
the host clock.

Prints one JSON line (rank 0).  ``--impl reference`` times the FP64 CPU oracle
instead, on the same workload.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import math
import os
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "ELT-SCAO frame latency p50/p99 µs + RMS jitter; MVM HBM GB/s vs peak"
FALLBACK_HBM_GBS = 6800.0
L2_FLUSH_BYTES = 512 << 20
BATCH = 100


def parse_args(argv=None):
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10000)
    ap.add_argument("--warmup", type=int, default=50)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--store", choices=["f32", "bf16", "f16", "fp8", "int8"], default="f32")
    ap.add_argument("--no-variants", action="store_true")
    ap.add_argument("--predictor", action="store_true",
                    help="the timed controller runs the learned slope predictor")
    ap.add_argument("--no-loop", action="store_true")
    # the persistent-loop runs of the serving sizing: 100,000 frames each, paced at 1 kHz
    # and flat out (p99.9 over 1e5 frames rests on 100 samples)
    ap.add_argument("--loop-frames", type=int, default=100000)
    ap.add_argument("--band-frames", type=int, default=2000)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--cpu-sample-s", type=float, default=15.0)
    ap.add_argument("--reference-budget-s", type=float, default=150.0)
    ap.add_argument("--oracle-worker", default=None, help=argparse.SUPPRESS)
    return ap.parse_args(argv)


# --------------------------------------------------------------------------- helpers
def pct(xs, q):
    s = sorted(xs)
    if not s:
        return float("nan")
    k = (len(s) - 1) * q
    lo, hi = int(math.floor(k)), int(math.ceil(k))
    return s[lo] + (s[hi] - s[lo]) * (k - lo)


def stats_us(xs):
    n = len(xs)
    mean = sum(xs) / n
    var = sum((x - mean) ** 2 for x in xs) / max(1, n - 1)
    return {"p50": pct(xs, 0.5), "p99": pct(xs, 0.99), "p999": pct(xs, 0.999), "mean": mean,
            "rms_jitter": math.sqrt(var), "min": min(xs), "max": max(xs),
            "peak_to_peak": max(xs) - min(xs)}


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(p) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return FALLBACK_HBM_GBS, "fallback"


KERNEL_SOURCES = ("frame_kernel.cu", "mvm_stream.cu", "calib_cog.cu", "stream_mvm.cuh", "pixel.cuh", "pred_tile.cuh")


def kernel_source_digest():
    """sha256[:16] over the sources of a frame's kernels."""
    h = hashlib.sha256()
    for name in KERNEL_SOURCES:
        with open(os.path.join(ROOT, "paper_1805_07254_gb300", "csrc", name), "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:16]


def recorded_traffic(workload):
    """DRAM bytes per frame-kernel launch from an ncu capture of the current kernel
    sources, else None."""
    p = os.path.join(ROOT, "profiles", "dram_traffic.txt")
    if not os.path.exists(p):
        return None
    dig = kernel_source_digest()
    for line in open(p):
        parts = line.split()
        if len(parts) == 4 and not line.startswith("#") and parts[0] == "frame" \
                and parts[1] == workload and parts[2] == dig:
            return float(parts[3])
    return None


class ClockSampler:
    """nvidia-smi clocks and throttle reasons, sampled every 50 ms while running."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.path = None

    def start(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.Q}",
                 "--format=csv,noheader,nounits", "-lms", "50"],
                stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None
        time.sleep(0.15)

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        time.sleep(0.1)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        rows = []
        for line in open(self.path):
            f = [x.strip() for x in line.split(",")]
            if len(f) < 9:
                continue
            try:
                rows.append((float(f[1]), float(f[2]), f[5:9]))
            except ValueError:
                continue
        os.unlink(self.path)
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"], "samples": 0}
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for _, _, fl in rows for i, v in enumerate(fl) if v == "Active"})
        sm = sorted(r[0] for r in rows)
        return {"sm_mhz": sm[len(sm) // 2], "sm_max_mhz": max(r[1] for r in rows),
                "reasons": reasons, "samples": len(rows)}


# --------------------------------------------------------------------------- oracle (CPU)
def oracle_worker(path):
    """Child process: time the FP64 oracle frame by frame (single thread)."""
    import numpy as np
    from oracle import pipeline as P
    d = np.load(path)
    budget = float(d["budget_s"])
    max_frames = int(d["max_frames"])
    loop = P.Loop(d["M"], d["dark"], d["flat"], d["subaps"], int(d["npx"]), float(d["gain"]),
                  float(d["leak"]))
    frames = d["frames"]
    times = []
    t_start = time.perf_counter()
    k = 0
    while k < max_frames and (time.perf_counter() - t_start) < budget:
        raw = frames[k % frames.shape[0]]
        t0 = time.perf_counter_ns()
        loop.step(raw)
        times.append((time.perf_counter_ns() - t0) / 1e3)
        k += 1
    print(json.dumps({"times_us": times}))


def run_oracle(cfg, frames, dark, flat, M, budget_s, max_frames, threads=1):
    """Per-frame times (us) of the FP64 oracle in a child process whose BLAS and
    OpenMP pools have `threads` threads."""
    import numpy as np
    fd, path = tempfile.mkstemp(suffix=".npz")
    os.close(fd)
    np.savez(path, M=M, dark=dark, flat=flat, subaps=cfg.subaps, npx=cfg.npx, gain=cfg.gain,
             leak=cfg.leak, frames=frames, budget_s=budget_s, max_frames=max_frames)
    env = dict(os.environ)
    for v in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS", "NUMEXPR_NUM_THREADS"):
        env[v] = str(threads)
    try:
        out = subprocess.run([sys.executable, os.path.abspath(__file__), "--oracle-worker", path],
                             capture_output=True, text=True, env=env, timeout=budget_s + 300)
    finally:
        os.unlink(path)
    if out.returncode != 0:
        raise RuntimeError("oracle worker failed: " + out.stderr[-2000:])
    return json.loads(out.stdout.strip().splitlines()[-1])["times_us"]


# --------------------------------------------------------------------------- workload
def make_workload(n_frames, store, cfg=None):
    import numpy as np
    import synth
    cfg = cfg or synth.elt_scao()
    frames, _ = synth.make_frames(cfg, 0, n_frames)
    dark, flat = synth.calibration_maps(cfg)
    M = synth.control_matrix(cfg).numpy()
    return cfg, frames.numpy(), dark.numpy(), flat.numpy(), np.ascontiguousarray(M)


def workload_config(cfg, store, info=None, predictor=False):
    c = {"workload": f"{cfg.name} ({cfg.frame_side}x{cfg.frame_side} u16 frame, "
                     f"{cfg.n_valid} subaps x {cfg.npx}x{cfg.npx} px, {cfg.nact}x{cfg.nslopes} "
                     f"{store} control matrix, {'learned slope predictor, ' if predictor else ''}"
                     f"leaky integrator)",
         "frame": f"{cfg.frame_side}x{cfg.frame_side}", "n_valid_subaps": cfg.n_valid,
         "nslopes": cfg.nslopes, "nact": cfg.nact, "matrix_store": store,
         "l2": f"flushed between timed steps (read of a {L2_FLUSH_BYTES >> 20} MiB device buffer, outside the events)"}
    if info:
        c["launch"] = {"slices": info["slices"], "blocks": info["blocks"],
                       "tile_rows": info["tile_rows"], "ring_stages": info["ring_stages"]}
    return c


# --------------------------------------------------------------------------- our arm
def time_steps(torch, r, d_frames, d_dm, flush, st, n_steps, n_warm, fused=True):
    """Per-step device times (us) from CUDA events on stream st.

    fused: one rtc_process_frame_async call per step (a frame's kernels);
    returns (step,).  Otherwise the two stage calls with an event between them;
    returns (pixel stage, reconstruction, step)."""
    E = torch.cuda.Event
    nF = len(d_frames)
    flush_out = torch.empty((), dtype=flush.dtype, device=flush.device)
    nev = 2 if fused else 3

    def one(i, ev):
        torch.sum(flush, dim=0, out=flush_out)
        if ev:
            ev[0].record(st)
        if fused:
            r.process_frame_async(d_frames[i % nF], d_dm, stream=st)
        else:
            r.centroid_async(d_frames[i % nF], stream=st)
            if ev:
                ev[1].record(st)
            r.reconstruct_async(None, d_dm, stream=st)
        if ev:
            ev[-1].record(st)

    with torch.cuda.stream(st):
        for i in range(n_warm):
            one(i, None)
        st.synchronize()
        evs = [tuple(E(enable_timing=True) for _ in range(nev)) for _ in range(n_steps)]
        for b0 in range(0, n_steps, BATCH):
            nb = min(BATCH, n_steps - b0)
            torch.cuda._sleep(int(2e6))          # device head start while the host enqueues
            for i in range(b0, b0 + nb):
                one(i, evs[i])
        st.synchronize()
    r.synchronize(st)                            # raises if a bounded device wait expired
    step = [evs[i][0].elapsed_time(evs[i][-1]) * 1e3 for i in range(n_steps)]
    if fused:
        return (step,)
    cog = [evs[i][0].elapsed_time(evs[i][1]) * 1e3 for i in range(n_steps)]
    mvm = [evs[i][1].elapsed_time(evs[i][2]) * 1e3 for i in range(n_steps)]
    return cog, mvm, step


def launch_floor(torch, flush, st, n_steps, n_warm=20):
    """Event time (us, p50) of one trivial kernel (a 1-element add) timed exactly
    like a frame: after the same L2 flush, between two events on st, queued behind
    a device sleep.  Every per-launch time above contains this much launch cost."""
    E = torch.cuda.Event
    tiny = torch.zeros(1, device=flush.device)
    flush_out = torch.empty((), dtype=flush.dtype, device=flush.device)
    with torch.cuda.stream(st):
        for _ in range(n_warm):
            torch.sum(flush, dim=0, out=flush_out)
            tiny.add_(1.0)
        st.synchronize()
        evs = [(E(enable_timing=True), E(enable_timing=True)) for _ in range(n_steps)]
        for b0 in range(0, n_steps, BATCH):
            torch.cuda._sleep(int(2e6))
            for i in range(b0, min(b0 + BATCH, n_steps)):
                torch.sum(flush, dim=0, out=flush_out)
                evs[i][0].record(st)
                tiny.add_(1.0)
                evs[i][1].record(st)
        st.synchronize()
    return pct([a.elapsed_time(b) * 1e3 for a, b in evs], 0.5)


def e2e_entry(s_launch, s_res, resident_headline, info, cfg, n, step_in_bytes, l2_bytes):
    """The e2e object: rtc_process_frame with pinned host buffers, synchronous, host
    clock.  Two modes of the same call: the call's own kernel launches (L2 flushed
    before each call) and the resident kernel (rtc_resident_start; no flush possible).  The
    resident figure is the headline when the step's inputs exceed L2.  (The mode's label
    is older than the second kernel of a frame; readers of the line know it by that.)"""
    launch = {"p50_us": round(s_launch["p50"], 3), "p99_us": round(s_launch["p99"], 3),
              "rms_jitter_us": round(s_launch["rms_jitter"], 3), "l2": "flushed before each call"}
    res = {"p50_us": round(s_res["p50"], 3), "p99_us": round(s_res["p99"], 3),
           "rms_jitter_us": round(s_res["rms_jitter"], 3),
           "l2": f"not flushed (step inputs {step_in_bytes / 1e6:.1f} MB against L2 {l2_bytes / 1e6:.1f} MB)"}
    head = s_res if resident_headline else s_launch
    return {"value": round(head["p50"], 3), "unit": "us", "p99_us": round(head["p99"], 3),
            "rms_jitter_us": round(head["rms_jitter"], 3),
            "mode": "resident kernel" if resident_headline else "one launch per call",
            "h2d_bytes_per_step": info["frame_bytes"], "d2h_bytes_per_step": 4 * cfg.nact,
            "steps": n, "launch_per_call": launch, "resident": res}


def matrix_l2_label(matrix_bytes, forced_stream):
    """How the loop's matrix stream meets L2: "resident" (at most 80 MB with the default
    policy: it stays in L2 from frame to frame), or "streamed" (evict_first)."""
    if forced_stream:
        return "streamed (evict_first; lines may still hit L2)"
    return "resident" if matrix_bytes <= (80 << 20) else "streamed (evict_first, larger than L2)"


def loop_entry(st_l, l2_label):
    """One persistent-loop run as a bench entry (latencies in us)."""
    return {"frames": int(st_l["frames"]), "frames_per_s": round(st_l["frames_per_s"], 1),
            "matrix_l2": l2_label,
            "e2e_p50_us": round(st_l["e2e_p50_us"], 2), "e2e_p99_us": round(st_l["e2e_p99_us"], 2),
            "e2e_p999_us": round(st_l["e2e_p999_us"], 2),
            "e2e_rms_jitter_us": round(st_l["e2e_rms_jitter_us"], 3),
            "e2e_p2p_us": round(st_l["e2e_p2p_us"], 2),
            "dev_p50_us": round(st_l["dev_p50_us"], 2), "dev_p99_us": round(st_l["dev_p99_us"], 2),
            "dev_p999_us": round(st_l["dev_p999_us"], 2),
            "dev_rms_jitter_us": round(st_l["dev_rms_jitter_us"], 3)}


REPLICA_STATS = ("p50", "p99", "p999", "rms_jitter", "peak_to_peak", "mean")


def reduce_replicas(torch, dist, stats, device):
    """Replicas (one controller per GPU): every latency statistic becomes its maximum
    over the ranks (the worst replica), frames/s the sum of the ranks' 1e6 / mean.
    dist is torch.distributed with a process group, or None for one rank."""
    vals = [float(stats[k]) for k in REPLICA_STATS]
    fps = 1e6 / float(stats["mean"])
    if dist is not None:
        t = torch.tensor(vals, device=device, dtype=torch.float64)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        f = torch.tensor([fps], device=device, dtype=torch.float64)
        dist.all_reduce(f, op=dist.ReduceOp.SUM)
        vals, fps = t.tolist(), float(f[0])
    return dict(zip(REPLICA_STATS, vals)), fps


def ours(args):
    import numpy as np
    import torch
    import torch.distributed as dist

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        dist.init_process_group("nccl", device_id=dev)

    from paper_1805_07254_gb300 import Rtc

    n_frames = 16
    cfg, frames, dark, flat, M = make_workload(n_frames, args.store)
    hbm_peak, peak_kind = measured_peaks()
    flush = torch.zeros(L2_FLUSH_BYTES // 4, dtype=torch.float32, device=dev)
    st = torch.cuda.Stream(device=dev)
    d_frames = [torch.from_numpy(frames[k]).contiguous().to(dev) for k in range(n_frames)]
    d_dm = torch.empty(cfg.nact, dtype=torch.float32, device=dev)

    def controller(store):
        r = Rtc(cfg.nsub, cfg.npx, cfg.nact, obs=cfg.obs, gain=cfg.gain, leak=cfg.leak,
                device=local)
        r.load_calib(dark, flat)
        r.load_cmat(M, store=store)
        return r

    # the predictor's weights do not change the timing
    from synth.mlp_init import init_mlp_params, flatten
    pred_params = flatten(init_mlp_params(0))
    r = controller(args.store)
    if args.predictor:
        r.load_predictor(pred_params, 0.3)
        r.set_predictor(True)
    info = r.info()

    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    sampler = ClockSampler(local)
    sampler.start()
    t_wall = time.perf_counter()
    (step,) = time_steps(torch, r, d_frames, d_dm, flush, st, args.steps, args.warmup, fused=True)
    t_wall = time.perf_counter() - t_wall
    clocks = sampler.stop()
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()

    # the same frames through the two stage kernels, for the per-stage split
    n_stage = min(args.steps, 2000)
    cog, mvm, step2 = time_steps(torch, r, d_frames, d_dm, flush, st, n_stage, args.warmup, fused=False)

    s_step, s_mvm, s_cog, s_step2 = stats_us(step), stats_us(mvm), stats_us(cog), stats_us(step2)
    mvm_bytes = info["matrix_bytes"] + 4 * info["nslopes"] + 8 * cfg.nact
    step_bytes = mvm_bytes + info["frame_bytes"] + info["calib_bytes"]
    frame_gbs = step_bytes / (s_step["mean"] * 1e-6) / 1e9
    mvm_gbs = mvm_bytes / (s_mvm["mean"] * 1e-6) / 1e9

    # e2e: the synchronous host-buffer C call, pinned frame in, DM commands out
    pin_frames = [torch.from_numpy(frames[k]).pin_memory() for k in range(n_frames)]
    pin_dm = torch.empty(cfg.nact, dtype=torch.float32).pin_memory()
    n_e2e = min(args.steps, 2000)
    e2e_us = []
    flush_out = torch.empty((), dtype=torch.float32, device=dev)
    for i in range(args.warmup + n_e2e):
        torch.sum(flush, dim=0, out=flush_out)
        torch.cuda.synchronize()
        t0 = time.perf_counter_ns()
        r.process_frame(pin_frames[i % n_frames], dm_out=pin_dm)
        t1 = time.perf_counter_ns()
        if i >= args.warmup:
            e2e_us.append((t1 - t0) / 1e3)
    s_e2e = stats_us(e2e_us)

    # the same call with the persistent kernel resident (rtc_resident_start): no kernel
    # launch per frame.  Nothing else may run on the GPU meanwhile, so there is no L2
    # flush between these calls; they are the headline e2e only when the step's inputs
    # are larger than L2 (the FP32 frame: 144.8 MB), as the timing rule requires
    r.resident_start()
    res_us = []
    try:
        for i in range(args.warmup + n_e2e):
            t0 = time.perf_counter_ns()
            r.process_frame(pin_frames[i % n_frames], dm_out=pin_dm)
            t1 = time.perf_counter_ns()
            if i >= args.warmup:
                res_us.append((t1 - t0) / 1e3)
    finally:
        r.resident_stop()
    s_res = stats_us(res_us)
    step_in_bytes = info["matrix_bytes"] + info["frame_bytes"] + info["calib_bytes"]
    l2_bytes = int(getattr(torch.cuda.get_device_properties(dev), "L2_cache_size", 0) or (126 << 20))
    resident_headline = step_in_bytes > l2_bytes

    variants = {}
    if not args.no_variants:
        for store in ("f32", "bf16", "f16", "fp8", "int8"):
            if store == args.store:
                continue
            rv = controller(store)
            iv = rv.info()
            (s2,) = time_steps(torch, rv, d_frames, d_dm, flush, st, min(args.steps, 2000),
                               args.warmup, fused=True)
            _, m2, _ = time_steps(torch, rv, d_frames, d_dm, flush, st, min(args.steps, 1000),
                                  args.warmup, fused=False)
            sv, mv = stats_us(s2), stats_us(m2)
            mb = iv["matrix_bytes"] + 4 * iv["nslopes"] + 8 * cfg.nact
            fb = mb + iv["frame_bytes"] + iv["calib_bytes"]
            variants[store] = {"p50_us": round(sv["p50"], 3), "p99_us": round(sv["p99"], 3),
                               "p999_us": round(sv["p999"], 3),
                               "rms_jitter_us": round(sv["rms_jitter"], 3),
                               "frame_hbm_gbs": round(fb / (sv["mean"] * 1e-6) / 1e9, 1),
                               "frame_frac_of_peak": round(fb / (sv["mean"] * 1e-6) / 1e9 / hbm_peak, 4),
                               "stage_mvm_us_mean": round(mv["mean"], 3),
                               "stage_mvm_hbm_gbs": round(mb / (mv["mean"] * 1e-6) / 1e9, 1)}
            rv.close()

    # reduced precision + learned predictor: BF16 matrix, predictor on (pixel stage,
    # prediction with the streaming reconstruction, and the sum: three kernels); the
    # weights do not change the timing
    if not args.no_variants:
        rp = controller("bf16")
        rp.load_predictor(pred_params, 0.3)
        rp.set_predictor(True)
        (s3,) = time_steps(torch, rp, d_frames, d_dm, flush, st, min(args.steps, 2000),
                           args.warmup, fused=True)
        sp = stats_us(s3)
        variants["bf16_predictor"] = {"p50_us": round(sp["p50"], 3), "p99_us": round(sp["p99"], 3),
                                      "p999_us": round(sp["p999"], 3),
                                      "rms_jitter_us": round(sp["rms_jitter"], 3),
                                      "kernels_per_frame": 3}
        rp.close()

    # stress sizing: six ELT WFS into one 4421 x 47664 FP8 matrix
    stress = None
    if not args.no_variants:
        import synth
        cfg6, frames6, dark6, flat6, M6 = make_workload(8, "fp8", synth.elt_scao_6wfs())
        r6 = Rtc(cfg6.nsub, cfg6.npx, cfg6.nact, n_wfs=cfg6.n_wfs, obs=cfg6.obs, gain=cfg6.gain,
                 leak=cfg6.leak, device=local)
        r6.load_calib(dark6, flat6)
        r6.load_cmat(M6, store="fp8")
        del M6
        i6 = r6.info()
        d_frames6 = [torch.from_numpy(frames6[k]).contiguous().to(dev) for k in range(8)]
        (s6,) = time_steps(torch, r6, d_frames6, d_dm, flush, st, min(args.steps, 2000),
                           args.warmup, fused=True)
        q6 = stats_us(s6)
        b6 = i6["matrix_bytes"] + 4 * i6["nslopes"] + 8 * cfg6.nact + i6["frame_bytes"] + i6["calib_bytes"]
        st6 = st6k = None
        if not args.no_loop:
            st6, _, _ = r6.run_loop(args.loop_frames, rate_hz=0.0, frames=frames6)
            st6k, _, _ = r6.run_loop(args.loop_frames, rate_hz=1000.0, frames=frames6)
        stress = {"workload": f"6 x {cfg6.frame_side}x{cfg6.frame_side} u16 frames, {cfg6.n_wfs * cfg6.n_valid} "
                              f"subaps, {cfg6.nact}x{i6['nslopes']} fp8 matrix + row scales",
                  "p50_us": round(q6["p50"], 3), "p99_us": round(q6["p99"], 3),
                  "p999_us": round(q6["p999"], 3), "rms_jitter_us": round(q6["rms_jitter"], 3),
                  "frame_hbm_gbs": round(b6 / (q6["mean"] * 1e-6) / 1e9, 1),
                  "frame_frac_of_peak": round(b6 / (q6["mean"] * 1e-6) / 1e9 / hbm_peak, 4)}
        for key, st_l in (("loop_max", st6), ("loop_1kHz", st6k)):
            if st_l:
                stress[key] = loop_entry(st_l, matrix_l2_label(i6["matrix_bytes"], 0))
        r6.close()
        del d_frames6

    # persistent real-time loop (rtc_run_loop): frames published by a host thread into
    # pinned mapped memory, DM commands back in host memory; paced at 1 kHz and flat
    # out, args.loop_frames frames each.  A matrix of at most 80 MB stays in L2 from
    # frame to frame ("resident"); the BF16 "evict_first" run streams it with that L2
    # policy instead.
    loop = {}
    if not args.no_loop:
        for store, pred, mode, rate, l2 in (("f32", False, "1kHz", 1000.0, 0),
                                            ("f32", False, "max", 0.0, 0),
                                            ("bf16", False, "max", 0.0, 0),
                                            ("bf16", False, "max", 0.0, 1),
                                            ("fp8", False, "max", 0.0, 0),
                                            ("bf16", True, "1kHz", 1000.0, 0),
                                            ("bf16", True, "max", 0.0, 0)):
            rl = controller(store)
            if pred:
                rl.load_predictor(pred_params, 0.3)
                rl.set_predictor(True)
            st_l, _, _ = rl.run_loop(args.loop_frames, rate_hz=rate, frames=frames[:8], matrix_l2=l2)
            key = f"{store}{'_predictor' if pred else ''}_{mode}{'_evict_first' if l2 else ''}"
            loop[key] = loop_entry(st_l, matrix_l2_label(rl.info()["matrix_bytes"], l2))
            rl.close()
        # a rolling readout at 1 kHz: 74 bands of 10 pixel rows (one row of
        # subapertures each), 10 us apart, so the last pixel arrives 730 us after
        # the first; latency from the last band's publication.  Equal slices, then
        # the asymmetric allocation for that readout (rtc_set_readout).
        bands, band_us = cfg.nsub, 10.0
        for store in ("f32", "bf16", "fp8"):
            rl = controller(store)
            for cut in (False, True):
                if cut:
                    rl.set_readout(bands, band_us)
                st_l, _, _ = rl.run_loop(args.band_frames, rate_hz=1000.0, frames=frames[:8],
                                         bands=bands, band_interval_us=band_us)
                loop[f"{store}_1kHz_{bands}bands_{'cut' if cut else 'equal'}"] = {
                    "frames": int(st_l["frames"]), "slices": rl.info()["slices"],
                    "band_interval_us": band_us,
                    "last_pixel_e2e_p50_us": round(st_l["e2e_p50_us"], 2),
                    "last_pixel_e2e_p99_us": round(st_l["e2e_p99_us"], 2),
                    "last_pixel_e2e_rms_jitter_us": round(st_l["e2e_rms_jitter_us"], 3),
                    "last_pixel_dev_p50_us": round(st_l["dev_p50_us"], 2),
                    "last_pixel_dev_p99_us": round(st_l["dev_p99_us"], 2),
                    "last_pixel_dev_rms_jitter_us": round(st_l["dev_rms_jitter_us"], 3)}
            rl.close()

    # replicas: the worst replica's latency statistics, the aggregate frames/s
    worst, total_fps = reduce_replicas(torch, dist if world > 1 else None, s_step, dev)
    value = worst["p50"]

    cpu = cpu_all = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        times = run_oracle(cfg, frames[:4], dark, flat, M, args.cpu_sample_s, 400)
        cpu = {"value": round(pct(times, 0.5), 1), "unit": "us", "cores": 1, "kind": "oracle",
               "sample": f"{len(times)} ELT frames through the FP64 oracle (single thread, "
                         f"time-bounded at {args.cpu_sample_s:.0f} s); p50 per frame"}
        # the same oracle with every host core in its BLAS pool (context for the single-thread
        # baseline: the 281 MB FP64 matrix-vector product is host-memory-bound)
        ncores = os.cpu_count() or 1
        times_mt = run_oracle(cfg, frames[:4], dark, flat, M, args.cpu_sample_s / 2, 400, threads=ncores)
        cpu_all = {"value": round(pct(times_mt, 0.5), 1), "unit": "us", "cores": ncores, "kind": "oracle",
                   "sample": f"{len(times_mt)} ELT frames through the FP64 oracle with {ncores} BLAS "
                             f"threads (time-bounded at {args.cpu_sample_s / 2:.0f} s); p50 per frame"}

    traffic = recorded_traffic(f"elt_{args.store}{'_pred' if args.predictor else ''}")
    floor_us = launch_floor(torch, flush, st, min(args.steps, 1000))
    line = {
        "metric": METRIC, "value": round(value, 3), "unit": "us", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": round(s_step["mean"] / 1e3, 6), "higher_is_better": False,
        "scaling": "weak", "vs_baseline": None, "dtype": args.store, "data": "synthetic",
        "config": workload_config(cfg, args.store, info, args.predictor),
        "p50_us": round(worst["p50"], 3), "p99_us": round(worst["p99"], 3),
        "p999_us": round(worst["p999"], 3), "rms_jitter_us": round(worst["rms_jitter"], 3),
        "peak_to_peak_us": round(worst["peak_to_peak"], 3), "mean_us": round(worst["mean"], 3),
        "frames_per_s": round(total_fps, 1),
        "stage_path_us_p50": {"calib_cog_kernel": round(s_cog["p50"], 3),
                              "mvm_stream_kernel": round(s_mvm["p50"], 3),
                              "step_two_kernels": round(s_step2["p50"], 3)},
        "stage_mvm_hbm_gbs": round(mvm_gbs, 1),
        "roofline": {"kernel": "frame_kernel + mvm_reduce_kernel", "bound": "hbm", "achieved": round(frame_gbs, 1),
                     "peak": hbm_peak, "peak_kind": peak_kind, "unit": "GB/s",
                     "frac": round(frame_gbs / hbm_peak, 4), "traffic": traffic,
                     "algorithmic_bytes": step_bytes,
                     "launch_floor_us": round(floor_us, 3)},
        "e2e": e2e_entry(s_e2e, s_res, resident_headline, info, cfg, n_e2e, step_in_bytes, l2_bytes),
        # (pixels and partials, sum; the predictor has a pixel stage of its own)
        "gpu_launches": args.steps * (3 if args.predictor else 2),
        "clocks": clocks,
        "timed_wall_s_incl_flush": round(t_wall, 3),
        "variants": variants,
        "stress_6wfs_fp8": stress,
        "loop": loop,
        "cpu_baseline": cpu,
        "cpu_baseline_all_cores": cpu_all,
    }
    if rank == 0:
        print(json.dumps(line), flush=True)
    r.close()
    if world > 1:
        dist.destroy_process_group()


# --------------------------------------------------------------------------- reference arm
def reference(args):
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    if rank != 0:
        return
    cfg, frames, dark, flat, M = make_workload(4, args.store)
    from oracle import quant as Q
    Ms = Q.stored_matrix(M, args.store).astype("float32") if args.store != "f32" else M
    want = args.warmup + args.steps
    times = run_oracle(cfg, frames, dark, flat, Ms, args.reference_budget_s, want)
    timed = times[args.warmup:] if len(times) > args.warmup else times
    s = stats_us(timed)
    line = {
        "impl": "reference", "metric": METRIC, "value": round(s["p50"], 1), "unit": "us",
        "n_gpus": world, "steps": len(timed), "warmup": min(args.warmup, len(times)),
        "ms_per_step": round(s["mean"] / 1e3, 3), "higher_is_better": False, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": workload_config(cfg, args.store),
        "p99_us": round(s["p99"], 1), "rms_jitter_us": round(s["rms_jitter"], 1),
        "cpu_baseline": {"value": round(s["p50"], 1), "unit": "us", "cores": 1, "kind": "oracle",
                         "sample": f"{len(timed)} of the {args.steps} requested frames "
                                   f"(time-bounded at {args.reference_budget_s:.0f} s), "
                                   "single-threaded FP64 oracle"},
        "e2e": {"value": round(s["p50"], 1), "unit": "us", "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


def main():
    args = parse_args()
    if args.oracle_worker:
        oracle_worker(args.oracle_worker)
        return
    if args.impl == "reference":
        reference(args)
    else:
        ours(args)


if __name__ == "__main__":
    main()
