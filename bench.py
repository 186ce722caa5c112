"""Throughput benchmark of the GB300 optical-flow velocimetry estimator.

python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Workload (one "step"): a time-resolved stream of 1001 synthetic 1024x1024
12-bit particle frames (0.08 particles/px, FWHM 2-3 px, 1 % noise, Rankine
vortex R 32 px / 3 px peak plus a uniform (1.3, -0.7) px shift), i.e. 1000
image pairs, each turned into a dense displacement field with 3 pyramid
levels (PSL 2), window radius 4 and 3 Gauss-Newton iterations per level,
FP32 storage, fused kernels, through ofv_compute_sequence.  The frames
(2 GB) are resident in HBM and larger than L2, so every pair reads its
inputs from DRAM.  Metric: velocity fields per second (whole job) and
Mvectors/s.  Extra lines of the same JSON object report 4 Mp and 21 Mp
streams, the FP16-storage path and the plain multi-kernel FP32 path.

Under torchrun every rank processes its own 1000-pair stream on its own GPU
(independent pairs: weak scaling, no collective on the data path); the
timing is the max over ranks.

--impl reference times the FP64 CPU oracle (test infrastructure) on the host
cores on a bounded sample of the same workload.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import math
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "velocity fields/s (Hz) and Mvectors/s at 1/4/21 Mp; % of HBM roofline"
H1, W1, FRAMES1 = 1024, 1024, 1001
FALLBACK_HBM_GBS = 6800.0


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=30)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-sizes", action="store_true", help="skip the 4 Mp / 21 Mp / variant lines")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--frames", type=int, default=FRAMES1, help="frames in the 1 Mp stream (pairs + 1)")
    ap.add_argument("--backward-only", action="store_true",
                    help="time only the reverse mode on 1 Mp pairs of the stream (one JSON line)")
    ap.add_argument("--batched-only", action="store_true",
                    help="time only the 64 uneven pairs through ofv_compute_batched (one JSON line)")
    ap.add_argument("--paper-only", action="store_true",
                    help="time only the paper's benchmark parameters (u8, NR 2, KR 10, IT 3) at 1 Mp (one JSON line)")
    return ap.parse_args()


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return FALLBACK_HBM_GBS, "fallback"


# ---------------------------------------------------------------------------
# clocks during the timed region
# ---------------------------------------------------------------------------
class ClockSampler:
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.file = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
        self.proc = None
        self.gpu = gpu_index

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.gpu}", f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=self.file, stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None
        time.sleep(0.25)

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        time.sleep(0.25)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.file.flush()
        self.file.seek(0)
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in self.file.read().splitlines():
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            for n, val in zip(names, parts[5:9]):
                if val.lower().startswith("active"):
                    reasons.add(n)
        os.unlink(self.file.name)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


def workload_config(nframes: int, ws: int) -> dict:
    """The headline workload, named the same way on both arms."""
    N = H1 * W1
    npairs = nframes - 1
    return {"workload": f"1024x1024 u16 12-bit Rankine+shift stream of {nframes} frames ({npairs} pairs), "
                        "PSL2 KR4 IT3, FP32 storage, fused kernels, ofv_compute_sequence",
            "pairs_total": npairs * ws, "pairs_per_rank": npairs, "parallelism": f"replicas{ws}",
            "l2": f"inputs ({nframes * N * 2 / 1e9:.2f} GB of frames) larger than L2" if nframes * N * 2 > 129e6
            else "inputs smaller than L2"}


# ---------------------------------------------------------------------------
# reference arm: the FP64 oracle on the host cores
# ---------------------------------------------------------------------------
def run_reference(args, ws, rank):
    if rank != 0:
        return
    import oracle
    import synth
    oracle.build()
    frames = synth.stream_frames(H1, W1, 2 + args.warmup + args.steps, seed=2)
    p = oracle.Params(psl=2, kr=4, it=3, bits=12)
    f64 = [f.astype(np.float64) for f in frames]
    for k in range(args.warmup):
        oracle.flow(f64[k], f64[k + 1], p)
    t0 = time.perf_counter()
    for k in range(args.steps):
        j = args.warmup + k
        oracle.flow(f64[j], f64[j + 1], p)
    dt = time.perf_counter() - t0
    value = args.steps / dt
    cores = oracle.num_threads()
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": "fields/s",
        "n_gpus": ws, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": 1e3 * dt / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": dict(workload_config(args.frames, ws),
                       step="one image pair of the stream (a bounded sample of it: the oracle at FP64)"),
        "cpu_baseline": {"value": value, "unit": "fields/s", "cores": cores, "kind": "oracle",
                         "sample": f"{args.steps} pairs of the 1 Mp stream, FP64, OpenMP over rows"},
        "e2e": {"value": value, "unit": "fields/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


# ---------------------------------------------------------------------------
# our arm
# ---------------------------------------------------------------------------
KERNEL_SOURCES = ("k_walk.cuh", "k_block.cuh", "k_block_inst.cuh", "iter_math.cuh", "ofv_common.cuh")


def kernel_source_hash():
    """Hash of the iteration kernel's sources with comments and blank lines
    removed: it changes when the code changes or a source is missing, not when
    a comment does."""
    import re
    h = hashlib.sha256()
    for f in KERNEL_SOURCES:
        path = os.path.join(ROOT, "paper_2509_25924_gb300", "csrc", f)
        if not os.path.exists(path):
            h.update(f"{f} is missing".encode())
            continue
        with open(path) as fh:
            src = re.sub(r"/\*.*?\*/", "", fh.read(), flags=re.S)
        lines = (re.sub(r"//.*$", "", ln).rstrip() for ln in src.splitlines())
        h.update("\n".join(ln for ln in lines if ln).encode())
    return h.hexdigest()[:16]


def ncu_record(workload: str) -> dict:
    """The committed ncu figures of the fused iteration kernel (DRAM bytes
    per launch, issue-active fraction), if they were taken on the current
    kernel source, else {}."""
    path = os.path.join(ROOT, "profiles", "traffic.json")
    try:
        with open(path) as f:
            d = json.load(f)
        e = d.get(workload)
        if e and e.get("kernel_hash") == kernel_source_hash():
            return e
    except Exception:
        pass
    return {}


def reduce_max(x: float, dist=None, device="cpu") -> float:
    """Max of a per-rank value over all ranks (the job's time is the slowest
    rank's); x itself without a process group."""
    if dist is None:
        return x
    import torch
    t = torch.tensor([x], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_rate(units_per_rank: int, ws: int, seconds_max: float) -> float:
    """Units all ranks processed over the slowest rank's time (weak scaling:
    every rank runs its own stream of the same size)."""
    return ws * units_per_rank / seconds_max


def run_ours(args, ws, rank, local):
    import torch
    import paper_2509_25924_gb300 as ofv
    import synth

    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    dist = None
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)

    def barrier():
        if dist is not None:
            dist.barrier()
        torch.cuda.synchronize()

    def max_over_ranks(x: float) -> float:
        return reduce_max(x, dist, dev)

    stream = torch.cuda.current_stream()
    nframes = args.frames
    frames_h = synth.stream_frames(H1, W1, nframes, seed=2)
    frames = torch.from_numpy(frames_h).to(dev)
    npairs = nframes - 1
    N = H1 * W1
    u = torch.empty((npairs, H1, W1), dtype=torch.float32, device=dev)
    v = torch.empty_like(u)
    params = ofv.ofv_default_params()
    h = ofv.ofv_create(H1, W1, params)

    def step():
        ofv.ofv_compute_sequence(h, nframes, frames, N * 2, u, v, N, stream)

    # nvidia-smi starts before the warm-up: its first queries (NVML start-up)
    # can hold up CUDA calls of this process for tens of ms, which must not
    # fall into the timed steps; its samples cover warm-up and timed steps
    sampler = ClockSampler(local)
    sampler.start()
    for _ in range(max(args.warmup, 0)):
        step()
    torch.cuda.synchronize()

    barrier()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(args.steps):
        step()
    e1.record(stream)
    torch.cuda.synchronize()
    barrier()
    clocks = sampler.stop()
    ms_total = max_over_ranks(e0.elapsed_time(e1))
    ms_step = ms_total / args.steps
    value = whole_job_rate(npairs * args.steps, ws, ms_total / 1e3)

    # dominant kernel: its share of device time and its algorithmic bytes,
    # from one step timed launch by launch (CUDA events on the launching
    # stream; this pass runs the launches in order on the caller's stream)
    ofv.ofv_profile_enable(h, True)
    step()
    prof = {}
    for k, name in ((ofv.OFV_K_INGEST, "ingest"), (ofv.OFV_K_REDUCE, "reduce"), (ofv.OFV_K_ITERATE, "iterate")):
        prof[name] = ofv.ofv_profile_read(h, k)
    ofv.ofv_profile_enable(h, False)
    peak, peak_kind = peaks()
    ms_k, n_k, b_k = prof["iterate"]
    share = ms_k / sum(p[0] for p in prof.values())
    # the kernel's time inside the timed steps: its share of the device time
    # of a step applied to the measured step time (the group streams overlap
    # launches, so a launch's own events would count shared time twice)
    kernel_ms_step = share * ms_step
    achieved = b_k / (kernel_ms_step / 1e3) / 1e9
    achieved_serial = (b_k / n_k) / (ms_k / n_k / 1e3) / 1e9
    alg_bytes_field = sum(p[2] for p in prof.values()) / npairs
    workload = "1Mp_stream_fp32_fused"
    # the fused path launches one kernel per timed record (ingest, reduce, iteration)
    launches_per_step = sum(p[1] for p in prof.values())
    roofline = {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                "frac": achieved / peak, "traffic": ncu_record(workload).get("dram_bytes_per_launch_scaled"),
                "kernel": "k_iter_block (one Gauss-Newton iteration of one level, all pairs of a group)",
                "how": "algorithmic bytes of the step's iteration launches / (kernel share of device time x "
                       "measured ms_per_step)",
                "alg_bytes_per_launch": b_k / n_k, "launches_per_step": n_k,
                "kernel_ms_per_step": kernel_ms_step,
                "peak_kind": f"{peak_kind} hbm_gbs (copy, burst)",
                "share_of_step": share,
                "frac_serialised": achieved_serial / peak,
                "launch_ms_serialised": ms_k / n_k,
                "step_alg_bytes_per_field": alg_bytes_field,
                "step_frac": alg_bytes_field * (value / ws) / 1e9 / peak}
    issue = ncu_record(workload).get("issue_active_pct")
    if issue is not None:
        # what bounds the kernel in fact: the schedulers issue on this share
        # of cycles (ncu smsp__issue_active, level-0 launch)
        roofline["issue_active_frac"] = issue / 100.0

    line = {
        "metric": METRIC, "value": value, "unit": "fields/s", "n_gpus": ws, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms_step, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": workload_config(nframes, ws),
        "mvectors_per_s": value * N / 1e6,
        "gpu_launches": launches_per_step * args.steps,
        "roofline": roofline,
        "clocks": clocks,
        "serialised_ms_per_step": {k: p[0] for k, p in prof.items()},
    }

    # end to end through the host-pointer entry point
    if not args.no_e2e:
        line["e2e"] = e2e(args, ofv, torch, h, frames_h, dev, stream, barrier, max_over_ranks, ws)

    line["derived_1Mp"] = derived_rates(ofv, torch, u, v, H1, W1, npairs, stream)

    if not args.no_sizes:
        line["sizes"] = sizes(ofv, torch, synth, dev, stream, frames, u, v)
        line["live_21Mp"] = live_loop(ofv, torch, synth, dev, stream)
        line["live_21Mp_3lanes"] = live_loop(ofv, torch, synth, dev, stream, ring=9, lanes=3)
        line["live_21Mp_paper_params"] = live_loop(ofv, torch, synth, dev, stream, n_pairs=500, paper_params=True)
        line["variants_1Mp"] = variants(ofv, torch, synth, dev, stream, frames, u, v)
        line["paper_perf_set"] = paper_perf_set(ofv, torch, synth, dev, stream)
        line["batched_64_uneven"] = batched_uneven(ofv, torch, synth, dev, stream)
        line["backward_1Mp"] = backward_1mp(ofv, torch, frames, dev, stream)
        line["single_pair_1Mp"] = single_pair(ofv, torch, frames, dev, stream)

    ofv.ofv_destroy(h)
    del u, v, frames

    if rank == 0 and ws == 1 and not args.no_cpu:
        line["cpu_baseline"] = cpu_baseline(frames_h)
    elif rank == 0:
        line["cpu_baseline"] = None

    if rank == 0:
        print(json.dumps(line), flush=True)
    if dist is not None:
        dist.destroy_process_group()


def e2e(args, ofv, torch, h, frames_h, dev, stream, barrier, max_over_ranks, ws):
    """Same metric end to end through ofv_compute_sequence_host: the stream's
    frames are read from pinned host memory and every field is written back
    to pinned host memory inside the timed region (uploads, compute and
    downloads overlap on three streams)."""
    H, W = H1, W1
    N = H * W
    npairs = min(400, frames_h.shape[0] - 1)
    host_frames = torch.from_numpy(frames_h[:npairs + 1].view(np.int16)).pin_memory()
    hu = torch.empty((npairs, H, W), dtype=torch.float32).pin_memory()
    hv = torch.empty_like(hu).pin_memory()

    def run():
        ofv.ofv_compute_sequence_host(h, npairs + 1, host_frames, N * 2, hu, hv, N, stream)

    # no clock sampler here: its NVML queries stalled single host-timed steps
    # of this leg (28 -> 42..74 ms); the device-resident leg records the clocks
    for _ in range(max(args.warmup, 1)):  # the same W warm-up steps as the device-resident leg
        run()
    torch.cuda.synchronize()
    # 20 steps (about 0.55 s): single steps of this host-timed leg are
    # sometimes held up for tens of ms (seen as 69 and 79 ms against 27 ms,
    # with no sampler running), and a longer window weighs such a stall
    # by its share of the sustained run
    steps = max(1, min(args.steps, 20))
    barrier()
    t0 = time.perf_counter()
    c0 = time.process_time()
    step_ms = []
    for _ in range(steps):
        ts = time.perf_counter()
        run()
        torch.cuda.synchronize()
        step_ms.append(1e3 * (time.perf_counter() - ts))
    dt = max_over_ranks(time.perf_counter() - t0)
    cpu_s = time.process_time() - c0
    value = ws * npairs * steps / dt
    out = {"value": value, "unit": "fields/s", "h2d_bytes_per_step": (npairs + 1) * N * 2,
           "d2h_bytes_per_step": npairs * N * 8, "pairs_per_step": npairs, "steps": steps,
           "api": "ofv_compute_sequence_host (host wall clock incl. H2D of every frame and D2H of every field)",
           "step_ms": step_ms, "host_cpu_s": cpu_s, "wall_s": dt}
    # context: one ofv_compute_host call per pair (both frames up, field down, one stream)
    hp = min(100, npairs)
    ring = 8
    pu = torch.empty((ring, H, W), dtype=torch.float32).pin_memory()
    pv = torch.empty_like(pu).pin_memory()

    def pairwise():
        for k in range(hp):
            ofv.ofv_compute_host(h, host_frames[k], host_frames[k + 1], pu[k % ring], pv[k % ring], stream)

    pairwise()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    pairwise()
    torch.cuda.synchronize()
    out["pairwise_ofv_compute_host_fields_per_s"] = hp / (time.perf_counter() - t0)
    # context: the host link itself (pinned copies of the fields buffer,
    # one direction at a time); the e2e rate follows it from box to box
    dbuf = torch.empty(hu.numel() // 4, dtype=torch.float32, device=dev)
    hbuf = hu.view(-1)[:dbuf.numel()]
    for name, fn in (("pinned_h2d_gbs", lambda: dbuf.copy_(hbuf, non_blocking=True)),
                     ("pinned_d2h_gbs", lambda: hbuf.copy_(dbuf, non_blocking=True))):
        with torch.cuda.stream(stream):
            fn()
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            for _ in range(3):
                fn()
            torch.cuda.synchronize()
        out[name] = 3 * dbuf.numel() * 4 / (time.perf_counter() - t0) / 1e9
    del dbuf
    return out


def time_sequence(ofv, torch, h, frames, n_frames, H, W, u, v, stream, reps, in_bytes=2):
    N = H * W
    npairs = n_frames - 1
    ofv.ofv_compute_sequence(h, n_frames, frames, N * in_bytes, u, v, N, stream)
    torch.cuda.synchronize()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(reps):
        ofv.ofv_compute_sequence(h, n_frames, frames, N * in_bytes, u, v, N, stream)
    e1.record(stream)
    torch.cuda.synchronize()
    return npairs * reps / (e0.elapsed_time(e1) / 1e3)


def field_error(torch, synth, fld, u, v, H, W, dev, inside=None, margin=16):
    """Mean and 99th percentile of |V - V_true| over the fields u, v (n x H x
    W, device) against the analytic displacement fld, at least `margin` px
    from the border and outside the body (inside(x, y) true)."""
    tu, tv = fld.grid(H, W)
    keep = np.zeros((H, W), bool)
    keep[margin:H - margin, margin:W - margin] = True
    if inside is not None:
        yy, xx = np.mgrid[0:H, 0:W].astype(np.float64)
        keep &= ~inside(xx, yy)
    k = torch.from_numpy(keep).to(dev)
    tu = torch.from_numpy(tu.astype(np.float32)).to(dev)
    tv = torch.from_numpy(tv.astype(np.float32)).to(dev)
    e = torch.hypot(u - tu, v - tv)[:, k].flatten()
    smp = e[torch.randint(0, e.numel(), (1 << 22,), device=dev)]
    return {"err_mean_px": float(e.mean()), "err_p99_px": float(torch.quantile(smp, 0.99))}


def sizes(ofv, torch, synth, dev, stream, frames1, u1, v1):
    out = {}
    cases = [("1Mp", 1024, 1024, None), ("4Mp", 2048, 2048, "turb"), ("21Mp", 4096, 5120, "wake")]
    for name, H, W, kind in cases:
        inside = None
        if kind is None:
            frames, nf, reps, u, v = frames1, min(101, frames1.shape[0]), 5, u1, v1
            fld = synth.stream_field(H, W)
        else:
            if kind == "turb":
                fld = synth.turbulence_field(H, W, seed=3).sampled(H, W)
                nf, reps = 33, 5
                fr = synth.stream_frames(H, W, nf, seed=3, ppp=0.1, field=fld, field_max=8.0)
            else:
                fld, inside = synth.wake_field(H, W)
                nf, reps = 9, 4
                fr = synth.stream_frames(H, W, nf, seed=4, ppp=0.1, field=fld, field_max=8.0, exclude=inside)
            frames = torch.from_numpy(fr).to(dev)
            u = torch.empty((nf - 1, H, W), dtype=torch.float32, device=dev)
            v = torch.empty_like(u)
        res = {}
        for label, kw in (("fused_fp32", {}), ("fused_fp16", {"storage": ofv.OFV_STORE_F16}),
                          ("fused_bf16", {"storage": ofv.OFV_STORE_BF16}),
                          ("plain_fp32", {"path": ofv.OFV_PATH_PLAIN})):
            h = ofv.ofv_create(H, W, ofv.ofv_default_params(**kw))
            try:
                fps = time_sequence(ofv, torch, h, frames, nf, H, W, u, v, stream, reps)
                ofv.ofv_profile_enable(h, True)
                ofv.ofv_compute_sequence(h, nf, frames, H * W * 2, u, v, H * W, stream)
                tot_b = 0.0
                it_ms, it_n, it_b = ofv.ofv_profile_read(h, ofv.OFV_K_ITERATE)
                for k in (ofv.OFV_K_INGEST, ofv.OFV_K_REDUCE, ofv.OFV_K_ITERATE):
                    tot_b += ofv.ofv_profile_read(h, k)[2]
                ofv.ofv_profile_enable(h, False)
                peak, _ = peaks()
                res[label] = {"fields_per_s": fps, "mvectors_per_s": fps * H * W / 1e6,
                              "step_frac_of_hbm": tot_b / (nf - 1) * fps / 1e9 / peak,
                              "iterate_kernel_frac_of_hbm": it_b / (it_ms / 1e3) / 1e9 / peak}
                if label != "plain_fp32":
                    torch.cuda.synchronize()
                    res[label].update(field_error(torch, synth, fld, u[:nf - 1], v[:nf - 1], H, W, dev, inside))
            finally:
                ofv.ofv_destroy(h)
        out[name] = res
        if kind is not None:
            del frames, u, v
            torch.cuda.empty_cache()
    return out


def single_pair(ofv, torch, frames, dev, stream, reps=50):
    """One 1 Mp pair at a time (no batching of pairs into a launch), three
    ways: ofv_compute on a handle, ofv_compute_noalloc (the library's fixed
    scratch array, image tiles staged by cp.async instead of TMA), and
    ofv_compute_strips with 2 strips run one after the other on this device
    (the layout a two-GPU split of one field uses, here without a second
    GPU).  Times with CUDA events over reps calls each."""
    H, W = H1, W1
    I1, I2 = frames[0], frames[1]
    u = torch.empty((H, W), device=dev)
    v = torch.empty_like(u)
    p = ofv.ofv_default_params()
    h = ofv.ofv_create(H, W, p)
    out = {}
    try:
        calls = {"ofv_compute": lambda: ofv.ofv_compute(h, I1, I2, u, v, stream),
                 "ofv_compute_noalloc": lambda: ofv.ofv_compute_noalloc(H, W, p, None, I1, I2, u, v, stream),
                 "ofv_compute_strips_2": lambda: ofv.ofv_compute_strips(h, 2, 8, I1, I2, u, v, stream)}
        for name, fn in calls.items():
            fn()
            torch.cuda.synchronize()
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            for _ in range(reps):
                fn()
            e1.record(stream)
            torch.cuda.synchronize()
            ms = e0.elapsed_time(e1) / reps
            out[name] = {"ms_per_pair": ms, "fields_per_s": 1e3 / ms}
    finally:
        ofv.ofv_destroy(h)
    out["workload"] = "the first pair of the 1 Mp stream (u16, PSL 2, KR 4, IT 3, FP32), one pair per call"
    return out


def derived_rates(ofv, torch, u, v, H, W, n, stream, reps=5):
    """Vorticity and recirculation-area count (Sec. 7, Eq. 6) over the n
    fields of the stream, resident in HBM: fields/s and the fraction of the
    measured copy bandwidth (algorithmic bytes: u, v read and omega written,
    12 B/px; u read, 4 B/px)."""
    N = H * W
    omega = torch.empty_like(u)
    counts = torch.empty(n, dtype=torch.int64, device=u.device)
    peak, _ = peaks()
    out = {}
    for name, fn, bpp in (("vorticity", lambda: ofv.ofv_vorticity(H, W, n, u, v, N, omega, stream), 12.0),
                          ("recirculation_area", lambda: ofv.ofv_recirculation_area(H, W, n, u, N, None, counts,
                                                                                   stream), 4.0)):
        fn()
        torch.cuda.synchronize()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(reps):
            fn()
        e1.record(stream)
        torch.cuda.synchronize()
        sec = e0.elapsed_time(e1) / 1e3 / reps
        out[name] = {"fields_per_s": n / sec, "gbs": n * N * bpp / sec / 1e9, "frac_of_hbm": n * N * bpp / sec / 1e9 / peak}
    del omega, counts
    return out


def variants(ofv, torch, synth, dev, stream, frames, u, v, n_frames=201, reps=5):
    """The estimator variants on the first n_frames of the 1 Mp stream:
    fields/s and the error against the analytic displacement of the stream
    (Rankine vortex plus uniform shift), mean and 99th percentile of |V -
    V_true| over pixels at least 16 px from the border, over the last 100
    pairs.  Warm start d: pair k starts from pair k-d's field."""
    H, W = H1, W1
    tu, tv = synth.stream_field(H, W).grid(H, W)
    tu = torch.from_numpy(tu.astype(np.float32)).to(dev)
    tv = torch.from_numpy(tv.astype(np.float32)).to(dev)
    cases = [
        ("box_direct_psl2_it3", {}),
        ("gauss_sigma2_psl2_it3", dict(window=ofv.OFV_WINDOW_GAUSS, window_sigma=2.0)),
        ("increment_psl2_it3", dict(increment_form=1)),
        ("warm_d8_psl2_it3", dict(warm_start=8)),
        ("warm_d8_psl0_it2", dict(warm_start=8, levels_psl=0, iterations=2)),
        ("warm_d8_psl0_it1", dict(warm_start=8, levels_psl=0, iterations=1)),
        ("warm_d1_psl0_it2", dict(warm_start=1, levels_psl=0, iterations=2)),
        ("warm_d16_psl0_it2", dict(warm_start=16, levels_psl=0, iterations=2)),
        ("warm_d16_psl2_it3", dict(warm_start=16)),
        ("cold_psl0_it2", dict(levels_psl=0, iterations=2)),
        ("mask_disk_psl2_it3", dict(mask="disk")),
    ]
    yy, xx = np.mgrid[0:H, 0:W]
    disk = ((xx - 700) ** 2 + (yy - 380) ** 2 >= 90 ** 2).astype(np.uint8)  # a 180 px masked disk
    out = {}
    s = (slice(None), slice(16, H - 16), slice(16, W - 16))
    for name, kw in cases:
        kw = dict(kw)
        mask = kw.pop("mask", None)
        h = ofv.ofv_create(H, W, ofv.ofv_default_params(**kw))
        try:
            if mask is not None:
                ofv.ofv_set_mask(h, torch.from_numpy(disk).to(dev), stream)
            rate = time_sequence(ofv, torch, h, frames, n_frames, H, W, u, v, stream, reps)
            k0 = n_frames - 1 - 100
            err = torch.hypot(u[k0:n_frames - 1][s] - tu[s[1:]], v[k0:n_frames - 1][s] - tv[s[1:]]).flatten()
            err = err[~err.isnan()]  # masked pixels have no vector
            smp = err[torch.randint(0, err.numel(), (1 << 22,), device=dev, generator=None)]
            out[name] = {"fields_per_s": rate, "err_mean_px": float(err.mean()),
                         "err_p99_px": float(torch.quantile(smp, 0.99))}
        finally:
            ofv.ofv_destroy(h)
    out["stream"] = (f"first {n_frames} frames of the 1 Mp bench stream, KR 4, FP32 storage, fused path; "
                     "defaults PSL 2 IT 3 unless named; error over the last 100 pairs (valid pixels only "
                     "with the mask: a 180 px disk masked)")
    return out


def paper_perf_set(ofv, torch, synth, dev, stream, cases=None):
    """The paper's own benchmark parameters (8-bit input, NR 2, KR 10, IT 3,
    PSL 0/1/2) on synthetic 8-bit particle streams at 1, 4, 10 and 21 Mp, for
    context beside its published rates (other hardware).  The paper gives no
    dimensions for its 10 Mp images; 5120 x 2048 is the 21 Mp camera's full
    width at half height."""
    out = {}
    for name, H, W, nf in cases or (("1Mp", 1024, 1024, 41), ("4Mp", 2048, 2048, 17), ("10Mp", 2048, 5120, 9),
                                    ("21Mp", 4096, 5120, 9)):
        fr = synth.stream_frames(H, W, nf, seed=7, ppp=0.05, bits=8).astype(np.uint8)
        frames = torch.from_numpy(fr).to(dev)
        u = torch.empty((nf - 1, H, W), dtype=torch.float32, device=dev)
        v = torch.empty_like(u)
        res = {}
        for psl in (0, 1, 2):
            p = ofv.ofv_default_params(input=ofv.OFV_IN_U8, bit_depth=8, norm_radius=2, kernel_radius=10,
                                       iterations=3, levels_psl=psl)
            h = ofv.ofv_create(H, W, p)
            try:
                res[f"psl{psl}_fields_per_s"] = time_sequence(ofv, torch, h, frames, nf, H, W, u, v, stream, 3,
                                                              in_bytes=1)
            finally:
                ofv.ofv_destroy(h)
        out[name] = res
        del frames, u, v
        torch.cuda.empty_cache()
    out["params"] = "u8 input, NR 2, KR 10, IT 3, PSL 0/1/2, FP32 storage, fused path, ofv_compute_sequence"
    return out


def live_loop(ofv, torch, synth, dev, stream, n_pairs=2000, ring=8, lanes=1, paper_params=False):
    """21 Mp live analogue: a device ring of `ring` pre-generated pairs of
    the cylinder-wake stream (5120x4096 u16), one CUDA graph per ring pair,
    replayed for n_pairs fields.  lanes = 1: one handle, graphs back to back
    on one stream.  lanes > 1: pair i runs on handle and stream i mod lanes,
    so consecutive fields overlap (each handle owns its workspace).  Per-field
    latency: CUDA events around each graph launch on its stream."""
    H, W = 4096, 5120
    fld, inside = synth.wake_field(H, W)
    if paper_params:  # the paper's benchmark parameters: 8-bit input, NR 2, KR 10, PSL 2, IT 3
        fr = synth.stream_frames(H, W, ring + 1, seed=4, ppp=0.1, bits=8, field=fld, field_max=8.0,
                                 exclude=inside).astype(np.uint8)
        params = dict(input=ofv.OFV_IN_U8, bit_depth=8, norm_radius=2, kernel_radius=10, levels_psl=2, iterations=3)
    else:
        fr = synth.stream_frames(H, W, ring + 1, seed=4, ppp=0.1, field=fld, field_max=8.0, exclude=inside)
        params = {}
    frames = torch.from_numpy(fr).to(dev)
    u = torch.empty((2 * lanes, H, W), dtype=torch.float32, device=dev)
    v = torch.empty_like(u)
    hs = [ofv.ofv_create(H, W, ofv.ofv_default_params(**params)) for _ in range(lanes)]
    streams = [stream] if lanes == 1 else [torch.cuda.Stream(device=dev) for _ in range(lanes)]
    graphs = []
    try:
        # graph of ring pair k on lane k mod lanes (ring is a multiple of lanes)
        for k in range(ring):
            ln = k % lanes
            graphs.append(ofv.ofv_graph_create(hs[ln], frames[k], frames[k + 1], u[2 * ln + (k // lanes) % 2],
                                               v[2 * ln + (k // lanes) % 2]))
        for k in range(ring):
            ofv.ofv_graph_launch(graphs[k], streams[k % lanes])
        torch.cuda.synchronize()
        e0 = [torch.cuda.Event(enable_timing=True) for _ in range(n_pairs)]
        e1 = [torch.cuda.Event(enable_timing=True) for _ in range(n_pairs)]
        start = torch.cuda.Event(enable_timing=True)
        end = torch.cuda.Event(enable_timing=True)
        start.record(stream)
        for st in streams:
            st.wait_event(start)
        for i in range(n_pairs):
            st = streams[i % lanes]
            e0[i].record(st)
            ofv.ofv_graph_launch(graphs[i % ring], st)
            e1[i].record(st)
        for st in streams:
            stream.wait_stream(st)
        end.record(stream)
        torch.cuda.synchronize()
        per = np.array([e0[i].elapsed_time(e1[i]) for i in range(n_pairs)])
        total = start.elapsed_time(end)
        # algorithmic bytes of one field (kernel timing pass of the same pipeline)
        ofv.ofv_profile_enable(hs[0], True)
        ofv.ofv_compute(hs[0], frames[0], frames[1], u[0], v[0], stream)
        field_bytes = sum(ofv.ofv_profile_read(hs[0], k)[2]
                          for k in (ofv.OFV_K_INGEST, ofv.OFV_K_REDUCE, ofv.OFV_K_ITERATE))
        ofv.ofv_profile_enable(hs[0], False)
        torch.cuda.synchronize()
    finally:
        for g in graphs:
            ofv.ofv_graph_destroy(g)
        for h in hs:
            ofv.ofv_destroy(h)
    del frames, u, v
    torch.cuda.empty_cache()
    kind = "u8, NR 2, KR 10, PSL 2, IT 3 (the paper's parameters)" if paper_params else "u16, PSL 2, KR 4, IT 3"
    return {"workload": f"5120x4096 cylinder-wake stream ({kind}), ring of {ring} pairs, one CUDA graph per pair, "
                        f"{lanes} handle/stream lane(s)",
            "pairs": n_pairs, "hz": n_pairs / (total / 1e3), "p50_ms": float(np.percentile(per, 50)),
            "p99_ms": float(np.percentile(per, 99)), "max_ms": float(per.max()),
            "frac_of_hbm": field_bytes * n_pairs / (total / 1e3) / 1e9 / peaks()[0]}


def batched_uneven(ofv, torch, synth, dev, stream, n_pairs=64, reps=5):
    """64 pairs with sizes drawn (seed 5) from {256^2, 512^2, 768x1024,
    1024^2}, turbulence displacement: one ofv_compute_batched call (one
    launch for all iterations) vs one ofv_compute per pair.  Each
    pair has its own device buffers; pairs of one size class share content."""
    classes = [(256, 256), (512, 512), (768, 1024), (1024, 1024)]
    rng = np.random.default_rng(5)
    pick = rng.integers(0, len(classes), size=n_pairs)
    content = {}
    for c in sorted(set(pick.tolist())):
        H, W = classes[c]
        fld = synth.turbulence_field(H, W, seed=3 + c).sampled(H, W)
        I1, I2 = synth.particle_pair(H, W, fld, ppp=0.1, dmin=2.0, dmax=3.0, seed=30 + c, noise=0.01,
                                     kind=synth.OUT_U16, field_max=8.0)
        content[c] = (torch.from_numpy(I1).to(dev), torch.from_numpy(I2).to(dev))
    pairs = []
    for c in pick.tolist():
        H, W = classes[c]
        a, b = content[c]
        pairs.append((a.clone(), b.clone(), torch.empty((H, W), device=dev), torch.empty((H, W), device=dev)))
    mpix = sum(p[0].numel() for p in pairs) / 1e6
    h = ofv.ofv_create(256, 256, ofv.ofv_default_params())
    try:
        ofv.ofv_compute_batched(h, pairs, stream)  # tunes on first use
        tune = ofv.ofv_batch_tuning(h)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for _ in range(reps):
            ofv.ofv_compute_batched(h, pairs, stream)
        torch.cuda.synchronize()
        batched = n_pairs * reps / (time.perf_counter() - t0)
        # the same batch recorded as a CUDA graph and replayed (no host work)
        g = ofv.ofv_graph_create_batched(h, pairs)
        try:
            ofv.ofv_graph_launch(g, stream)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            for _ in range(reps):
                ofv.ofv_graph_launch(g, stream)
            torch.cuda.synchronize()
            graph = n_pairs * reps / (time.perf_counter() - t0)
        finally:
            ofv.ofv_graph_destroy(g)
    finally:
        ofv.ofv_destroy(h)
    handles = {c: ofv.ofv_create(*classes[c], ofv.ofv_default_params()) for c in content}
    try:
        def seq():
            for c, p in zip(pick.tolist(), pairs):
                ofv.ofv_compute(handles[c], p[0], p[1], p[2], p[3], stream)
        seq()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for _ in range(reps):
            seq()
        torch.cuda.synchronize()
        sequential = n_pairs * reps / (time.perf_counter() - t0)
    finally:
        for hh in handles.values():
            ofv.ofv_destroy(hh)
    # reverse mode on the same pairs: dL/dI1, dL/dI2 and dL/dw of the 5x5
    # pre-filter for random dL/du, dL/dv (forward recomputed inside)
    bh = {c: ofv.ofv_create(*classes[c], ofv.ofv_default_params(prefilter=1)) for c in content}
    gen = torch.Generator(device=dev)
    gen.manual_seed(5)
    grads = {}
    for c in content:
        shp = classes[c]
        grads[c] = (torch.randn(shp, device=dev, generator=gen), torch.randn(shp, device=dev, generator=gen),
                    torch.empty(shp, device=dev), torch.empty(shp, device=dev), torch.empty(25, device=dev))
    torch.cuda.synchronize()
    try:
        def bwd():
            for c, p in zip(pick.tolist(), pairs):
                gu, gv, g1, g2, gw = grads[c]
                ofv.ofv_backward(bh[c], p[0], p[1], gu, gv, g1, g2, gw, stream)
        bwd()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for _ in range(reps):
            bwd()
        torch.cuda.synchronize()
        backward = n_pairs * reps / (time.perf_counter() - t0)
    finally:
        for hh in bh.values():
            ofv.ofv_destroy(hh)
    return {"pairs": n_pairs, "mpix_per_batch": mpix, "batched_fields_per_s": batched,
            "batched_graph_fields_per_s": graph,
            "batched_mvectors_per_s": batched * mpix / n_pairs, "sequential_fields_per_s": sequential,
            "backward_pairs_per_s": backward, "backward_mvectors_per_s": backward * mpix / n_pairs,
            "tuning": tune, "timing": "host wall clock over 5 batches, synchronised at the end (batched calls "
                                      "after the tuning one are asynchronous; the graph rate replays the "
                                      "recorded batch 5 times the same way)"}


def cpu_baseline(frames_h):
    import oracle
    oracle.build()
    p = oracle.Params(psl=2, kr=4, it=3, bits=12)
    a = frames_h[0].astype(np.float64)
    b = frames_h[1].astype(np.float64)
    oracle.flow(a, b, p)  # warm-up
    n = 0
    t0 = time.perf_counter()
    while True:
        oracle.flow(frames_h[n + 1].astype(np.float64), frames_h[n + 2].astype(np.float64), p)
        n += 1
        if time.perf_counter() - t0 > 8.0 or n >= 8:
            break
    dt = time.perf_counter() - t0
    return {"value": n / dt, "unit": "fields/s", "cores": oracle.num_threads(), "kind": "oracle",
            "sample": f"{n} pairs of the 1 Mp stream, FP64 oracle with OpenMP over rows "
                      f"({oracle.num_threads()} threads)"}


def backward_1mp(ofv, torch, frames, dev, stream, n_pairs=20, reps=3):
    """Reverse mode on 1 Mp pairs of the stream (12-bit, PSL 2, KR 4, IT 3,
    5x5 pre-filter on): dL/dI1, dL/dI2 and dL/dw for random dL/du, dL/dv,
    the forward pass recomputed inside; ms per pair by CUDA events.  Also
    with the paper's benchmark normalization (NR 2)."""
    N = H1 * W1
    gen = torch.Generator(device=dev)
    gen.manual_seed(11)
    gu = torch.randn((H1, W1), device=dev, generator=gen)
    gv = torch.randn((H1, W1), device=dev, generator=gen)
    g1 = torch.empty((H1, W1), device=dev); g2 = torch.empty_like(g1); gw = torch.empty(25, device=dev)

    def ms_per_pair(params):
        h = ofv.ofv_create(H1, W1, params)
        try:
            def run():
                for k in range(n_pairs):
                    ofv.ofv_backward(h, frames[k], frames[k + 1], gu, gv, g1, g2, gw, stream)
            run()
            torch.cuda.synchronize()
            e0 = torch.cuda.Event(enable_timing=True); e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            for _ in range(reps):
                run()
            e1.record(stream)
            torch.cuda.synchronize()
            return e0.elapsed_time(e1) / (reps * n_pairs)
        finally:
            ofv.ofv_destroy(h)

    ms = ms_per_pair(ofv.ofv_default_params(prefilter=1))
    ms_nr = ms_per_pair(ofv.ofv_default_params(prefilter=1, norm_radius=2))
    return {"ms_per_pair": ms, "pairs_per_s": 1e3 / ms, "mvectors_per_s": N / 1e3 / ms,
            "workload": "1024x1024 u16 stream pairs, PSL 2 KR 4 IT 3, pre-filter on; gradients w.r.t. both frames "
                        "and the 25 weights, forward recomputed",
            "nr2": {"ms_per_pair": ms_nr, "pairs_per_s": 1e3 / ms_nr,
                    "workload": "the same with local normalization NR 2 (the paper's benchmark value)"}}


def run_backward_only(args):
    import torch
    import paper_2509_25924_gb300 as ofv
    import synth
    dev = torch.device("cuda", 0)
    torch.cuda.set_device(dev)
    frames = torch.from_numpy(synth.stream_frames(H1, W1, 21, seed=2)).to(dev)
    print(json.dumps({"backward_1Mp": backward_1mp(ofv, torch, frames, dev, torch.cuda.current_stream(),
                                                   reps=max(1, args.steps))}), flush=True)


def main():
    args = parse()
    ws, rank, local = dist_env()
    if args.impl == "reference":
        run_reference(args, ws, rank)
        return
    if args.backward_only:
        run_backward_only(args)
        return
    if args.batched_only:
        import torch
        import paper_2509_25924_gb300 as ofv
        import synth
        dev = torch.device("cuda", 0)
        torch.cuda.set_device(dev)
        print(json.dumps({"batched_64_uneven": batched_uneven(ofv, torch, synth, dev, torch.cuda.current_stream())}),
              flush=True)
        return
    if args.paper_only:
        import torch
        import paper_2509_25924_gb300 as ofv
        import synth
        dev = torch.device("cuda", 0)
        torch.cuda.set_device(dev)
        print(json.dumps({"paper_perf_set": paper_perf_set(ofv, torch, synth, dev, torch.cuda.current_stream(),
                                                           cases=(("1Mp", 1024, 1024, 41),))}), flush=True)
        return
    run_ours(args, ws, rank, local)


if __name__ == "__main__":
    main()
