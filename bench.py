#!/usr/bin/env python
"""Benchmark: integral histograms of a 64-frame 1920x1080 sequence, 64 bins.

One step = one pass of the hot path over the 64 frames: the fused quantise +
2-D scan (rows a1-a5) of every frame in one persistent batched launch, and a
region query of 1000 rectangles per frame (row a6) in one launch.  ``value``
is frames/s with the frames already resident in HBM; the plain per-frame
form (64 launches of each kernel) is reported beside it.  ``e2e`` is the same
metric through ``ihist_batch_upload_compute`` (row a7): frames in pinned host
memory, uploaded on a copy stream, two 32-frame batches alternating so one
uploads while the other computes, query results copied back to the host --
all inside the timed region.

Usage: python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]
Under torchrun each rank is an independent replica on its own GPU with its
own frames (the work shards by frame; no collective on the data path); rank 0
prints one JSON line.  ``--impl reference`` times the CPU oracle instead.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "IH frames/s & written GB/s vs HBM peak; served p50/p99 vs plain per-frame launch"
H, W, NBINS, NFRAMES, NRECTS = 1080, 1920, 64, 64, 1000
SIGMA = 20.0
WORKLOAD = ("sequence of 64 frames 1920x1080 uint8, smooth gradient + Gaussian noise sigma=20 "
            "clipped to [0,255], B=64 uniform bins, uint32 bin-major output, 1000 region queries per frame")
PROFILE = os.path.join(ROOT, "profiles", "batch_kernel_64x1080p_b64.txt")
PROFILE_MP64 = os.path.join(ROOT, "profiles", "scan_kernel_8192x8192_b128.txt")
SCAN_SOURCES = ("ihist_scan.cuh", "ihist_device.cuh")


def parse_args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=("ours", "reference"))
    ap.add_argument("--e2e-steps", type=int, default=0, help="0 = min(steps, 30)")
    ap.add_argument("--cpu-seconds", type=float, default=12.0, help="oracle sample budget")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-configs", action="store_true",
                    help="skip the other workloads (640x480, uneven 256-frame batch, 8192x8192) "
                         "and the other bin structures (edges, joint RGB)")
    ap.add_argument("--layout", choices=("bin", "pixel", "quad"), default="bin",
                    help="output layout of the timed path (the workload's is bin-major; the others for captures)")
    ap.add_argument("--serve-seconds", type=float, default=10.0,
                    help="simulated seconds of the serving workload per server mode (0 = skip)")
    ap.add_argument("--frames", type=int, default=64,
                    help="frames per step (64 = the workload; smaller only for profiler captures)")
    ap.add_argument("--case", choices=("sequence", "mp64-slice", "query-slice", "vga"), default="sequence",
                    help="mp64-slice: only a few launches of the 8192x8192 x 128-bin scan's launch shape "
                         "on the top --slice-rows rows (a profiler capture of that kernel at a few GB); "
                         "query-slice: the plain and the row-bucketed region query of 2^18 rectangles on "
                         "the top 1024 rows of that frame (4 GiB of H); vga: the 640x480 x 32-bin "
                         "frames, ihist_compute + ihist_query of 1000 rectangles each, overlap=1, 64 "
                         "frames per step (the per-frame launches a profiler lists)")
    ap.add_argument("--slice-rows", type=int, default=768)
    return ap.parse_args()


def dist_env():
    return (int(os.environ.get("RANK", "0")), int(os.environ.get("WORLD_SIZE", "1")),
            int(os.environ.get("LOCAL_RANK", "0")))


def max_over_ranks(values, world: int, device=None) -> list:
    """Element-wise maximum of per-rank timings over all ranks: the slowest
    replica decides the job's time."""
    import torch
    t = torch.tensor([float(v) for v in values], dtype=torch.float64, device=device)
    if world > 1:
        import torch.distributed as dist
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return t.tolist()


def job_throughput(frames_per_rank: int, steps: int, world: int, elapsed_ms: float) -> float:
    """Frames per second of the whole job: every rank's frames over the slowest rank's time."""
    return world * frames_per_rank * steps / (elapsed_ms / 1000.0)


def make_frame(rank: int, f: int) -> np.ndarray:
    """Frame f of rank `rank`'s sequence: gradient plus N(0, 20^2) noise, its
    own substream of the workload's seed."""
    from paper_1711_01919_gb300 import synth
    return synth.gradient_frame(synth.substream_seed(synth.workload_seed(2), rank * 100000 + f), H, W, SIGMA)


def make_frames(rank: int, n: int = 0) -> np.ndarray:
    n = n or NFRAMES
    out = np.empty((n, H, W), dtype=np.uint8)
    for f in range(n):
        out[f] = make_frame(rank, f)
    return out


def make_rects() -> np.ndarray:
    from paper_1711_01919_gb300 import synth
    return synth.rects(synth.workload_seed(2) + 1, NRECTS, H, W)


def fnv1a64_of_hashes(hashes) -> int:
    """FNV-1a 64 over the little-endian bytes of a list of 64-bit frame hashes
    (one value for a set of frames)."""
    h = 0xCBF29CE484222325
    for v in hashes:
        for byte in int(v).to_bytes(8, "little"):
            h = ((h ^ byte) * 0x100000001B3) & 0xFFFFFFFFFFFFFFFF
    return h


def algorithmic_bytes_per_frame() -> int:
    return H * W * NBINS * 4 + H * W  # uint32 output written once + uint8 frame read once


def scan_source_hash() -> str:
    h = hashlib.sha256()
    for name in SCAN_SOURCES:
        with open(os.path.join(ROOT, "paper_1711_01919_gb300", "csrc", name), "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:16]


def profiled_traffic(path=PROFILE):
    """DRAM bytes per scan launch from a committed ncu summary, if it was
    taken on the current kernel source; else None."""
    try:
        kv = {}
        for line in open(path):
            if "=" in line and not line.lstrip().startswith("#"):
                k, v = line.split("#", 1)[0].split("=", 1)
                kv[k.strip()] = v.strip()
        if kv.get("scan_source_sha256_16") != scan_source_hash():
            return None
        return int(float(kv["traffic_bytes_per_launch"]))
    except (OSError, KeyError, ValueError):
        return None


def measured_peak():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return float(json.load(f)["hbm_gbs"]), "measured"
    except (OSError, KeyError, ValueError):
        return 6800.0, "fallback"


class _Nvml:
    """SM clock, power and clock-event reasons of one GPU read through NVML
    (the library nvidia-smi itself reads), for sampling every few
    milliseconds; None where NVML is missing."""

    REASONS = ((0x4, "sw_power_cap"), (0x8, "hw_slowdown"), (0x20, "sw_thermal_slowdown"),
               (0x40, "hw_thermal_slowdown"), (0x80, "hw_power_brake_slowdown"))

    def __init__(self, bus_id: str):
        import ctypes
        self.ct = ctypes
        self.lib = ctypes.CDLL("libnvidia-ml.so.1")
        if self.lib.nvmlInit_v2() != 0:
            raise OSError("nvmlInit failed")
        self.dev = ctypes.c_void_p()
        if self.lib.nvmlDeviceGetHandleByPciBusId_v2(bus_id.encode(), ctypes.byref(self.dev)) != 0:
            raise OSError("no NVML device at %s" % bus_id)
        self.reasons_fn = getattr(self.lib, "nvmlDeviceGetCurrentClocksEventReasons", None) or \
            self.lib.nvmlDeviceGetCurrentClocksThrottleReasons

    def sample(self):
        ct = self.ct
        clk, mx, mw, rs = ct.c_uint(0), ct.c_uint(0), ct.c_uint(0), ct.c_ulonglong(0)
        if self.lib.nvmlDeviceGetClockInfo(self.dev, 1, ct.byref(clk)) != 0:  # NVML_CLOCK_SM
            return None
        self.lib.nvmlDeviceGetMaxClockInfo(self.dev, 1, ct.byref(mx))
        self.lib.nvmlDeviceGetPowerUsage(self.dev, ct.byref(mw))
        self.reasons_fn(self.dev, ct.byref(rs))
        return clk.value, mx.value, mw.value / 1000.0, rs.value

    def close(self):
        self.lib.nvmlShutdown()


class ClockSampler:
    """Clocks and throttle reasons during a timed region: NVML every 5 ms in
    a thread (a timed region of 0.1 s still gets ~20 samples) and nvidia-smi
    every 200 ms as a cross-check."""

    FIELDS = ("index,pci.bus_id,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, nvml_bus_id: str | None = None, period_s: float = 0.005):
        self.proc = None
        self.path = os.path.join(tempfile.gettempdir(), "ihist_clocks_%d.csv" % os.getpid())
        self.period_s = period_s
        self.nvml_bus_id = nvml_bus_id
        self.nvml_rows = []
        self.thread = None

    def start(self):
        try:
            self.fh = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", "--query-gpu=" + self.FIELDS, "--format=csv,noheader,nounits",
                                          "-lms", "200"], stdout=self.fh, stderr=subprocess.DEVNULL)
        except (OSError, ValueError):
            self.proc = None
        if self.nvml_bus_id:
            import threading
            try:
                nv = _Nvml(self.nvml_bus_id)
            except (OSError, AttributeError):
                return
            self.stop_flag = threading.Event()

            def loop():
                while not self.stop_flag.is_set():
                    r = nv.sample()
                    if r is not None:
                        self.nvml_rows.append(r)
                    time.sleep(self.period_s)
                nv.close()

            self.thread = threading.Thread(target=loop, daemon=True)
            self.thread.start()

    def _smi_rows(self, bus_id):
        if self.proc is None:
            return []
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.fh.close()
        allrows = []
        for line in open(self.path):
            parts = [p.strip() for p in line.split(",")]
            if len(parts) >= 10:
                allrows.append(parts)
        rows = [r for r in allrows if bus_id and r[1].lower().endswith(bus_id.lower())]
        if not rows and len({r[1] for r in allrows}) == 1:
            rows = allrows
        try:
            os.remove(self.path)
        except OSError:
            pass
        return rows

    def stop(self, bus_id: str | None):
        if self.thread is not None:
            self.stop_flag.set()
            self.thread.join(timeout=5)
        rows = self._smi_rows(bus_id)
        names = ("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap")
        smi_sm = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        smi_mx = [float(r[3]) for r in rows if r[3].replace(".", "").isdigit()]
        smi_reasons = {n for r in rows for n, v in zip(names, r[6:10]) if v.strip().lower() == "active"}
        if self.nvml_rows:
            sm = [float(r[0]) for r in self.nvml_rows]
            reasons = {n for r in self.nvml_rows for bit, n in _Nvml.REASONS if r[3] & bit} | smi_reasons
            return {"sm_mhz": statistics.median(sm), "sm_mhz_min": min(sm),
                    "sm_max_mhz": max(max(r[1] for r in self.nvml_rows), max(smi_mx, default=0.0)),
                    "reasons": sorted(reasons), "samples": len(self.nvml_rows),
                    "power_w_max": max(r[2] for r in self.nvml_rows),
                    "source": "NVML every %.0f ms during the timed region (+ %d nvidia-smi samples at 200 ms)"
                              % (1000 * self.period_s, len(rows))}
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        return {"sm_mhz": statistics.median(smi_sm) if smi_sm else None,
                "sm_max_mhz": max(smi_mx) if smi_mx else None,
                "reasons": sorted(smi_reasons), "samples": len(rows), "source": "nvidia-smi every 200 ms"}


def nvml_bus_id(dev):
    """PCI bus id of a torch device in NVML's form (domain:bus:device.0)."""
    import torch
    try:
        p = torch.cuda.get_device_properties(dev)
        return "%08x:%02x:%02x.0" % (p.pci_domain_id, p.pci_bus_id, p.pci_device_id)
    except AttributeError:
        return None


def cpu_baseline(frames: np.ndarray, seconds: float, threads: int) -> dict:
    """The CPU oracle (Algorithm 1) on a bounded sample of the frames."""
    import oracle
    out = np.empty((NBINS, H, W), dtype=np.uint32)
    done, t0 = 0, time.perf_counter()
    while done < len(frames) and (done == 0 or time.perf_counter() - t0 < seconds):
        if threads > 1:
            oracle.integral_histogram_threads(frames[done], NBINS, threads, out)
        else:
            oracle.integral_histogram(frames[done], NBINS, out)
        done += 1
    dt = time.perf_counter() - t0
    return {"value": done / dt, "unit": "frames/s", "cores": threads, "kind": "oracle",
            "sample": "%d of the %d frames (1920x1080, 64 bins), %s Algorithm 1 in C, %.1f s"
                      % (done, len(frames), "bins-parallel" if threads > 1 else "single-threaded", dt)}


def host_cores() -> int:
    try:
        return len(os.sched_getaffinity(0))
    except AttributeError:
        return os.cpu_count() or 1


def run_mp64_slice(args) -> int:
    """The 8192x8192 x 128-bin frame's scan launch shape (the tiling its plan
    resolves to) on a slice of the frame's top rows: the launches a profiler
    captures for that workload without holding 32 GiB on the device."""
    import torch

    from paper_1711_01919_gb300 import build as cuda_build
    from paper_1711_01919_gb300 import ihist, synth
    cuda_build.build()
    ihist.load()
    h, w, b = args.slice_rows, 8192, 128
    with ihist.Plan(8192, w, b) as full:
        tune = dict(full.tune)
    img = torch.from_numpy(synth.sinusoid_frame(synth.workload_seed(5), 8192, w)[:h].copy()).cuda()
    out = torch.empty((b, h, w), dtype=torch.int32, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    keep = {k: tune[k] for k in ("rows_per_band", "bins_per_cta", "chunks_per_warp", "groups_per_cta", "ctas_per_sm",
                                 "warps_per_cta")}
    with ihist.Plan(h, w, b, tune=keep) as plan:
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2 * (args.warmup + args.steps))]
        for k in range(args.warmup + args.steps):
            ev[2 * k].record()
            ihist.ihist_compute(plan.handle, img.data_ptr(), w, out.data_ptr(), s)
            ev[2 * k + 1].record()
        torch.cuda.synchronize()
        if plan.status() != ihist.IHIST_OK:
            raise SystemExit("device status error in the 8192-column slice")
        ms = [ev[2 * k].elapsed_time(ev[2 * k + 1]) for k in range(args.warmup, args.warmup + args.steps)]
        print(json.dumps({"case": "mp64-slice", "rows": h, "W": w, "B": b, "tile": tile_of(plan),
                          "full_frame_tile": tune, "launch_ms": ms,
                          "bytes_per_launch": h * w * b * 4 + h * w}), flush=True)
    return 0


def run_query_slice(args) -> int:
    """The two bin-major region queries (ihist_query, ihist_query_sorted with
    8 bins per pass) on the top 1024 rows of the 8192x8192 x 128-bin frame,
    2^18 random rectangles: the launches a profiler captures for the query's
    DRAM traffic at 4 GiB of H (more than 129 MB of L2, as at full size)."""
    import torch

    from paper_1711_01919_gb300 import build as cuda_build
    from paper_1711_01919_gb300 import ihist, synth
    cuda_build.build()
    ihist.load()
    h, w, b, n = 1024, 8192, 128, 1 << 18
    img = torch.from_numpy(synth.sinusoid_frame(synth.workload_seed(5), 8192, w)[:h].copy()).cuda()
    rects = torch.from_numpy(synth.rects(synth.workload_seed(5) + 1, n, h, w)).cuda()
    s = torch.cuda.current_stream().cuda_stream
    with ihist.Plan(h, w, b) as plan:
        out = plan.compute(img)
        q1 = torch.empty((n, b), dtype=torch.int32, device="cuda")
        q2 = torch.empty_like(q1)
        work = torch.empty((plan.query_work_bytes(n, 8),), dtype=torch.uint8, device="cuda")
        ms = {"plain": [], "sorted": []}
        for k in range(args.warmup + args.steps):
            for name in ("plain", "sorted"):
                a, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                if name == "plain":
                    ihist.ihist_query(plan.handle, out.data_ptr(), rects.data_ptr(), n, q1.data_ptr(), s)
                else:
                    ihist.ihist_query_sorted(plan.handle, out.data_ptr(), rects.data_ptr(), n, q2.data_ptr(), 8,
                                             work.data_ptr(), work.numel(), s)
                e.record()
                torch.cuda.synchronize()
                if k >= args.warmup:
                    ms[name].append(a.elapsed_time(e))
        if plan.status() != ihist.IHIST_OK or not torch.equal(q1, q2):
            raise SystemExit("query slice: device status error or the two queries differ")
        print(json.dumps({"case": "query-slice", "rows": h, "W": w, "B": b, "rects": n, "ms": ms}), flush=True)
    return 0


def run_vga(args) -> int:
    """64 frames of 640x480 with 32 bins per step, each ihist_compute (plan
    tune overlap=1) followed by ihist_query of 1000 rectangles, 8 inputs and
    8 outputs in rotation: the per-frame launch pairs of the 640x480
    workload, for a profiler's launch list and captures."""
    import torch

    from paper_1711_01919_gb300 import build as cuda_build
    from paper_1711_01919_gb300 import ihist, synth
    cuda_build.build()
    ihist.load()
    h, w, b = 480, 640, 32
    seed = synth.workload_seed(1)
    fr = [torch.from_numpy(synth.uniform_frame(synth.substream_seed(seed, i), h, w)).cuda() for i in range(8)]
    ou = [torch.empty((b, h, w), dtype=torch.int32, device="cuda") for _ in range(8)]
    rects = torch.from_numpy(synth.rects(seed + 1, 1000, h, w)).cuda()
    q = torch.empty((1000, b), dtype=torch.int32, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    us = []
    with ihist.Plan(h, w, b, tune={"overlap": 1}) as plan:
        for k in range(args.warmup + args.steps):
            a, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            a.record()
            for i in range(64):
                ihist.ihist_compute(plan.handle, fr[i % 8].data_ptr(), w, ou[i % 8].data_ptr(), s)
                ihist.ihist_query(plan.handle, ou[i % 8].data_ptr(), rects.data_ptr(), 1000, q.data_ptr(), s)
            e.record()
            torch.cuda.synchronize()
            if k >= args.warmup:
                us.append(a.elapsed_time(e) * 1e3 / 64)
        if plan.status() != ihist.IHIST_OK:
            raise SystemExit("vga case: device status error")
        print(json.dumps({"case": "vga", "H": h, "W": w, "B": b, "rects": 1000, "us_per_frame": us}), flush=True)
    return 0


def run_reference(args):
    rank, world, _ = dist_env()
    if rank != 0:
        return 0
    import oracle
    oracle.build()
    frames = make_frames(0, max(1, min(NFRAMES, args.steps + args.warmup)))
    cores = host_cores()
    out = np.empty((NBINS, H, W), dtype=np.uint32)
    for i in range(args.warmup):
        oracle.integral_histogram_threads(frames[i % len(frames)], NBINS, cores, out)
    times = []
    used = cores
    for i in range(args.steps):
        t0 = time.perf_counter()
        _, used = oracle.integral_histogram_threads(frames[(args.warmup + i) % len(frames)], NBINS, cores, out)
        times.append(time.perf_counter() - t0)
    total = sum(times)
    value = args.steps / total
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": "frames/s", "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1000.0 * total / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u32",
        "data": "synthetic",
        "config": {"workload": WORKLOAD, "frames_per_step": 1, "H": H, "W": W, "B": NBINS,
                   "layout": "bin-major", "step": "one frame (bounded sample of the 64-frame sequence)"},
        "cpu_baseline": {"value": value, "unit": "frames/s", "cores": used, "kind": "oracle",
                         "sample": "%d frames of the workload, one per step, bins-parallel Algorithm 1 in C"
                                   % args.steps},
        "e2e": {"value": value, "unit": "frames/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


def serving_report(seconds: float) -> dict:
    """Served p50/p99 per request class, continuous batching against plain
    per-frame launches, on the same Poisson request stream (frames of the
    uneven mix at 2000/s, queries of 10,000 rectangles at 200/s), two runs of
    each server pooled, and the frame throughput of both servers when the
    same requests arrive 1000x faster than they can be served."""
    from paper_1711_01919_gb300 import serve

    keep = ("completed", "rejected", "p50_ms", "p99_ms", "max_ms", "per_s", "launch_wait_p99_ms")
    out = {"workload": "Poisson arrivals for %.1f s: frames at 2000/s (320x240..1920x1080, 16-64 bins), "
                       "queries of 10,000 rects at 200/s and searches for a 64x64 patch (stride 8) at 50/s "
                       "against a random resident histogram; 40 GB budget, LRU eviction" % seconds}
    # a short discarded pass of each server first: the first seconds of a
    # process's first serving runs measured slower whichever server ran first
    # (frame p99 0.52-0.55 ms against 0.43 ms once both had run); then two
    # measured runs of each in the order batched, plain, plain, batched (the
    # run order alone moved p99 by ~5% between identical code paths), each
    # server's latencies pooled over its two runs
    import numpy as np
    for mode in ("batched", "plain"):
        serve.serve(mode=mode, duration_s=min(seconds, 2.0))
    runs = {"batched": [], "plain": []}
    for mode in ("batched", "plain", "plain", "batched"):
        runs[mode].append(serve.serve(mode=mode, duration_s=seconds))
    for mode, reps in runs.items():
        out[mode] = {"runs": len(reps)}
        for k in ("frame", "query", "search"):
            lat = np.concatenate([r[k]["latencies_ms"] for r in reps])
            out[mode][k] = {"completed": int(sum(r[k]["completed"] for r in reps)),
                            "rejected": int(sum(r[k]["rejected"] for r in reps)),
                            "p50_ms": float(np.percentile(lat, 50)), "p99_ms": float(np.percentile(lat, 99)),
                            "max_ms": float(lat.max()),
                            "per_s": float(np.mean([r[k]["per_s"] for r in reps])),
                            "p99_ms_per_run": [r[k]["p99_ms"] for r in reps],
                            "launch_wait_p99_ms_per_run": [r[k]["launch_wait_p99_ms"] for r in reps]}
        out[mode]["frame"]["by_path"] = [r["frame"]["by_path"] for r in reps]
        out[mode]["launch_sizes"] = [r["launch_sizes"] for r in reps]
        out[mode]["host_issue_p50_ms"] = reps[0]["host_issue_p50_ms"]
        out[mode]["evicted"] = [r["evicted"] for r in reps]
    for mode in ("batched", "plain"):
        rep = serve.serve(mode=mode, duration_s=seconds / 2, saturate=True)
        out["saturated_" + mode] = {"frames_per_s": rep["frame"]["per_s"], "frames": rep["frame"]["completed"],
                                    "frame_p99_ms": rep["frame"]["p99_ms"]}
    return out


def _time_ms(fn, stream, reps: int = 50, warm: int = 10) -> dict:
    """Median and min of `reps` CUDA-event timings of fn on `stream` after
    `warm` untimed runs, each bracketed by device synchronisations."""
    import torch
    for _ in range(warm):
        fn()
    ts = []
    for _ in range(reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record(stream)
        fn()
        b.record(stream)
        torch.cuda.synchronize()
        ts.append(a.elapsed_time(b))
    return {"median": statistics.median(ts), "min": min(ts)}


def _median_ms(fn, stream, reps: int = 50, warm: int = 10) -> float:
    return _time_ms(fn, stream, reps, warm)["median"]


def tile_of(plan):
    """The tiling a plan's frames run with, or the path that has none."""
    from paper_1711_01919_gb300 import ihist
    return "two launches (count, emit)" if ihist.two_launch_plan(plan.handle) else plan.tune


def configs_report(stream, peak: float) -> dict:
    """The other workloads of the method, each timed on its own (median and
    min of 50 after 10 warm-ups, CUDA events): one 640x480 frame with 32 bins and 1000
    queries per launch pair (8 frames and 8 outputs in rotation, 315 MB > L2);
    a 256-frame batch of uneven size (320x240 .. 1920x1080, 16/32/64 bins),
    default and autotuned (as live launches), the autotuned one
    also replayed from a captured CUDA graph; one 8192x8192 frame with 128
    bins (34.4 GB out) and 2^20 queries on it."""
    import torch

    from paper_1711_01919_gb300 import autotune, ihist, synth
    s = stream.cuda_stream
    rep = {}
    # 640x480, 32 bins, 1000 queries
    h, w, b = 480, 640, 32
    seed = synth.workload_seed(1)
    host_fr = [synth.uniform_frame(synth.substream_seed(seed, i), h, w) for i in range(8)]
    rep["input_fnv1a64"] = {"vga_640x480_frames": [hex(synth.fnv1a64_rows(x)) for x in host_fr]}
    fr = [torch.from_numpy(x).cuda() for x in host_fr]
    del host_fr
    ou = [torch.empty((b, h, w), dtype=torch.int32, device="cuda") for _ in range(8)]
    rects = torch.from_numpy(synth.rects(seed + 1, 1000, h, w)).cuda()
    q = torch.empty((1000, b), dtype=torch.int32, device="cuda")
    byts = 64 * (h * w * b * 4 + h * w)
    vga_tuned = autotune.tune_plan(h, w, b)
    for label, tune in (("vga_640x480_b32_1000q", None), ("vga_640x480_b32_1000q_overlapped", {"overlap": 1}),
                        ("vga_640x480_b32_1000q_autotuned", dict(vga_tuned, overlap=1))):
        with ihist.Plan(h, w, b, tune=tune) as plan:
            def vga():
                for i in range(64):
                    ihist.ihist_compute(plan.handle, fr[i % 8].data_ptr(), w, ou[i % 8].data_ptr(), s)
                    ihist.ihist_query(plan.handle, ou[i % 8].data_ptr(), rects.data_ptr(), 1000, q.data_ptr(), s)
            tm = _time_ms(vga, stream)
            ms = tm["median"]
            if plan.status() != ihist.IHIST_OK:
                raise SystemExit("device status error in the 640x480 run")
            rep[label] = {"frames_per_s": 64e3 / ms, "us_per_frame": ms * 1e3 / 64,
                          "us_per_frame_min": tm["min"] * 1e3 / 64,
                          "gbs": byts / ms / 1e6, "frac": byts / ms / 1e6 / peak,
                          "form": "ihist_compute + ihist_query per frame" + (", overlap=1" if tune else ""),
                          "tile": tile_of(plan)}
    del fr, ou, rects, q
    # 256 uneven frames in one launch
    specs = synth.uneven_batch_specs(synth.workload_seed(3), 256)
    host_fr = [synth.uniform_frame(sd, h, w) for (h, w, nb, sd) in specs]
    rep["input_fnv1a64"]["uneven_256_frames_combined"] = hex(fnv1a64_of_hashes(
        [synth.fnv1a64_rows(x) for x in host_fr]))
    fr = [torch.from_numpy(x).cuda() for x in host_fr]
    del host_fr
    ou = [torch.empty((nb, h, w), dtype=torch.int32, device="cuda") for (h, w, nb, sd) in specs]
    nbs = [nb for (h, w, nb, sd) in specs]
    byts = sum(h * w * nb * 4 + h * w for (h, w, nb, sd) in specs)
    entry = {"frames": 256, "algorithmic_bytes": byts, "form": "one ihist_batch_compute"}
    # the autotuner picks the layout (no queries in this workload) and, for
    # it, the launch shape
    auto_layout, auto_tune, layout_ms = autotune.tune_batch_layout([(h, w, nb) for (h, w, nb, sd) in specs], 0)
    names = {ihist.IHIST_BIN_MAJOR: "bin-major", ihist.IHIST_PIXEL_MAJOR: "pixel-major", ihist.IHIST_QUAD_MAJOR: "quad-major"}
    for label, tune, layout in (("default", None, ihist.IHIST_BIN_MAJOR), ("autotuned", auto_tune, auto_layout)):
        with ihist.Batch(fr, nbs, [layout] * len(fr), outs=ou, tune=tune or None) as batch:
            tm = _time_ms(batch.compute, stream)
            ms = tm["median"]
            if batch.status() != ihist.IHIST_OK:
                raise SystemExit("device status error in the uneven batch")
            entry[label] = {"ms": ms, "ms_min": tm["min"], "frames_per_s": 256e3 / ms, "gbs": byts / ms / 1e6,
                            "frac": byts / ms / 1e6 / peak, "items": batch.items(), "layout": names[layout],
                            "path": "two-launch" if ihist.two_launch_batch(batch.handle) else "look-back"}
            if label == "autotuned":
                entry[label]["tune"] = auto_tune
                entry[label]["layout_ms_while_tuning"] = {names[k]: v for k, v in layout_ms.items()}
                # captured once in a CUDA graph and replayed (the look-back kernel with that tiling)
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g):
                    batch.compute()
                gms = _median_ms(g.replay, stream)
                if batch.status() != ihist.IHIST_OK:
                    raise SystemExit("device status error in the graph replay")
                entry[label]["graph_replay_ms"] = gms
                entry[label]["graph_replay_frac"] = byts / gms / 1e6 / peak
    rep["uneven_256_batch"] = entry
    del fr, ou
    torch.cuda.empty_cache()
    # 8192 x 8192, 128 bins, 2^20 queries
    h = w = 8192
    b = 128
    host_img = synth.sinusoid_frame(synth.workload_seed(5), h, w)
    rep["input_fnv1a64"]["sinusoid_8192x8192"] = hex(synth.fnv1a64_rows(host_img))
    img = torch.from_numpy(host_img).cuda()
    del host_img
    out = torch.empty((b, h, w), dtype=torch.int32, device="cuda")
    rects = torch.from_numpy(synth.rects(synth.workload_seed(5) + 1, 1 << 20, h, w)).cuda()
    q = torch.empty((1 << 20, b), dtype=torch.int32, device="cuda")
    with ihist.Plan(h, w, b) as plan:
        clocks = ClockSampler(nvml_bus_id(torch.cuda.current_device()))
        clocks.start()
        tm = _time_ms(lambda: ihist.ihist_compute(plan.handle, img.data_ptr(), w, out.data_ptr(), s), stream)
        ms = tm["median"]
        clk = clocks.stop(None)
        tq = _time_ms(lambda: ihist.ihist_query(plan.handle, out.data_ptr(), rects.data_ptr(), 1 << 20,
                                                q.data_ptr(), s), stream)
        qms = tq["median"]
        sorted_ms = {}
        work = torch.empty((plan.query_work_bytes(1 << 20, 4),), dtype=torch.uint8, device="cuda")
        for bpp in (4, 8, 16):
            if work.numel() < plan.query_work_bytes(1 << 20, bpp):
                work = torch.empty((plan.query_work_bytes(1 << 20, bpp),), dtype=torch.uint8, device="cuda")
            q2 = torch.empty_like(q)
            sorted_ms[bpp] = _median_ms(lambda: ihist.ihist_query_sorted(
                plan.handle, out.data_ptr(), rects.data_ptr(), 1 << 20, q2.data_ptr(), bpp, work.data_ptr(),
                work.numel(), s), stream)
            if not torch.equal(q2, q):
                raise SystemExit("sorted and plain 8192x8192 queries differ")
            del q2
        del work
        if plan.status() != ihist.IHIST_OK:
            raise SystemExit("device status error in the 8192x8192 run")
        byts = h * w * b * 4 + h * w
        rep["mp64_8192x8192_b128"] = {"scan_ms": ms, "scan_ms_min": tm["min"], "gbs": byts / ms / 1e6, "frac": byts / ms / 1e6 / peak,
                                      "bytes_per_launch": byts, "traffic": profiled_traffic(PROFILE_MP64),
                                      "traffic_source": "ncu DRAM bytes of the same launch shape on the top rows "
                                                        "of the frame, scaled to 8192 rows (profiles/)",
                                      "clocks": clk, "query_ms_2p20_rects": qms, "query_ms_min": tq["min"],
                                      "query_sorted_ms_2p20_rects": {"bins_per_pass_%d" % k: v
                                                                     for k, v in sorted_ms.items()},
                                      "tile": tile_of(plan)}
        rep["mp64_8192x8192_b128"].update(query_gather_report(out, qms, 1 << 20, b, stream))
    del img, out, rects, q
    torch.cuda.empty_cache()
    rep["host_output_1080p_b64"] = host_output_report(stream, peak)
    rep["window_search_1080p_b64"] = window_search_report(stream)
    rep["paper_mappings_1080p_b64"] = mappings_report(stream, peak)
    return rep


def query_gather_report(hist, query_ms: float, nrects: int, nbins: int, stream) -> dict:
    """The random-gather ceiling of a bin-major region query: 2^26 random
    4-byte loads over the same 32 GiB histogram (torch.take), timed like the
    query.  A (rect, bin) pair of Eq. 2 needs four such loads, so the probe
    bounds the pairs per second any gather-per-corner kernel can reach."""
    import torch
    n = 1 << 26
    g = torch.Generator(device=hist.device)
    g.manual_seed(1711)
    idx = torch.randint(0, hist.numel(), (n,), device=hist.device, dtype=torch.int64, generator=g)
    flat = hist.view(-1)
    ms = _median_ms(lambda: torch.take(flat, idx), stream)
    del idx
    gathers_per_s = n / (ms / 1e3)
    pairs = nrects * nbins
    ceiling_ms = 4 * pairs / gathers_per_s * 1e3
    return {"gather_probe": {"loads": n, "ms": ms, "loads_per_s": gathers_per_s,
                             "form": "torch.take of 2^26 uniform random words of the 32 GiB histogram"},
            "query_pairs": pairs, "query_ms_at_gather_ceiling": ceiling_ms,
            "query_frac_of_gather_ceiling": ceiling_ms / query_ms,
            "query_algorithmic_gbs": pairs * 20 / (query_ms / 1e3) / 1e9}


def mappings_report(stream, peak: float) -> dict:
    """The paper's GPU mappings (CW-STS, CW-TiS, WF-TiS; comparison kernels
    built on this GPU) against the default plan and the fused look-back kernel,
    one 1080p frame with 64 bins each, same output, same algorithmic bytes."""
    import torch

    from paper_1711_01919_gb300 import ihist, synth
    s = stream.cuda_stream
    img = torch.from_numpy(synth.gradient_frame(synth.workload_seed(2), H, W)).cuda()
    out = torch.empty((NBINS, H, W), dtype=torch.int32, device="cuda")
    byts = algorithmic_bytes_per_frame()
    rep = {}
    for name, m in ihist.MAPPINGS.items():
        nb = ihist.ihist_mapping_workspace_bytes(m, H, W, NBINS)
        work = torch.empty((max(nb, 1),), dtype=torch.uint8, device="cuda")
        ms = _median_ms(lambda: ihist.ihist_mapping_compute(m, H, W, NBINS, img.data_ptr(), W, out.data_ptr(),
                                                            work.data_ptr() if nb else 0, s), stream)
        rep[name] = {"ms_per_frame": ms, "frames_per_s": 1e3 / ms, "frac": byts / ms / 1e6 / peak}
        del work
    # the default plan, and the fused look-back kernel at its default tiling;
    # then the same frame into the pixel-major layout [y][x][b]
    for suffix, layout in (("", ihist.IHIST_BIN_MAJOR), ("_pixel_major", ihist.IHIST_PIXEL_MAJOR)):
        for name, tune in (("default_plan", None), ("fused_look_back", {"ctas_per_sm": 32})):
            with ihist.Plan(H, W, NBINS, layout, tune=tune) as plan:
                ms = _median_ms(lambda: ihist.ihist_compute(plan.handle, img.data_ptr(), W, out.data_ptr(), s), stream)
                rep[name + suffix] = {"ms_per_frame": ms, "frames_per_s": 1e3 / ms, "frac": byts / ms / 1e6 / peak,
                                      "tile": tile_of(plan)}
    return rep


def window_search_report(stream) -> dict:
    """Sliding-window search over one resident 1080p histogram (64 bins):
    64x64 windows every 4 pixels (255 x 465 = 118,575 windows), each scored
    by histogram intersection with a target from Eq. 2's four lookups per
    bin, for both layouts of H."""
    import torch

    from paper_1711_01919_gb300 import ihist, synth
    img = synth.gradient_frame(synth.workload_seed(2), H, W)
    d = torch.from_numpy(img).cuda()
    target = torch.from_numpy(np.bincount(((img[500:564, 900:964].astype(np.int64) * NBINS) >> 8).ravel(),
                                          minlength=NBINS).astype(np.int32)).cuda()
    out = {}
    for name, layout in (("bin_major", ihist.IHIST_BIN_MAJOR), ("pixel_major", ihist.IHIST_PIXEL_MAJOR)):
        with ihist.Plan(H, W, NBINS, layout) as plan:
            hist = plan.compute(d)
            scores = plan.window_search(hist, target, 64, 64, 4)
            ms = _median_ms(lambda: plan.window_search(hist, target, 64, 64, 4, out=scores), stream)
            best = torch.zeros(1, dtype=torch.int64, device="cuda")
            bms = _median_ms(lambda: ihist.ihist_window_search(plan.handle, hist.data_ptr(), target.data_ptr(), 64, 64,
                                                               4, 0, best.data_ptr(), stream.cuda_stream), stream)
            if plan.status() != ihist.IHIST_OK:
                raise SystemExit("device status error in the window search")
            n = scores.numel()
            out[name] = {"ms": ms, "windows": n, "windows_per_s": n / ms * 1e3,
                         "corner_gbs": n * 4 * NBINS * 4 / ms / 1e6, "best_window_only_ms": bms}
        del hist
    return out


def host_output_report(stream, peak: float, n: int = 16) -> dict:
    """Stand-alone mode: the integral histogram of each 1080p frame written
    straight into page-locked host memory by the scan kernel (its stores
    cross the CPU-GPU link; no device copy of H, no separate transfer),
    against the rate of a plain device-to-host copy of the same bytes."""
    import torch

    from paper_1711_01919_gb300 import ihist, synth
    s = stream.cuda_stream
    seed = synth.workload_seed(2)
    fr = [torch.from_numpy(synth.gradient_frame(synth.substream_seed(seed, i), H, W)).cuda() for i in range(4)]
    host = [torch.empty((NBINS, H, W), dtype=torch.int32).pin_memory() for _ in range(2)]
    dev = torch.empty((NBINS, H, W), dtype=torch.int32, device="cuda")
    nb = H * W * NBINS * 4
    with ihist.Plan(H, W, NBINS) as plan:
        def run():
            for i in range(n):
                ihist.ihist_compute(plan.handle, fr[i % 4].data_ptr(), W, host[i % 2].data_ptr(), s)
        ms = _median_ms(run, stream, reps=3, warm=1) / n
        if plan.status() != ihist.IHIST_OK:
            raise SystemExit("device status error in the host-output run")
    copy_ms = _median_ms(lambda: host[0].copy_(dev, non_blocking=True), stream, reps=3, warm=1)
    return {"frames_per_s": 1e3 / ms, "ms_per_frame": ms, "link_gbs": nb / ms / 1e6,
            "d2h_copy_gbs": nb / copy_ms / 1e6, "frac_of_d2h_copy": copy_ms / ms,
            "form": "ihist_compute with d_out in page-locked host memory (bin-major)"}


def layouts_report(d_frames, outs, d_rects, stream, steps: int = 10) -> dict:
    """The bench step (one batched launch over the resident frames + one
    batched query launch) in each output layout, on the same frames and the
    same output memory."""
    import torch

    from paper_1711_01919_gb300 import ihist
    n = d_frames.shape[0]
    s = stream.cuda_stream
    flat = outs.view(-1)
    out = {}
    byts = n * (H * W * NBINS * 4 + H * W)
    for name, layout in (("bin-major", ihist.IHIST_BIN_MAJOR), ("pixel-major", ihist.IHIST_PIXEL_MAJOR),
                         ("quad-major", ihist.IHIST_QUAD_MAJOR)):
        o = flat.view((n,) + ihist.out_shape(H, W, NBINS, layout))
        q = torch.empty((n * NRECTS * NBINS,), dtype=torch.int32, device=flat.device)
        with ihist.Batch([d_frames[f] for f in range(n)], NBINS, [layout] * n, outs=[o[f] for f in range(n)]) as b:
            def step():
                ihist.ihist_batch_compute(b.handle, s)
                ihist.ihist_batch_query_all(b.handle, d_rects.data_ptr(), NRECTS, q.data_ptr(), s)

            for _ in range(3):
                step()
            ev = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
            torch.cuda.synchronize()
            ev[0].record(stream)
            for _ in range(steps):
                ihist.ihist_batch_compute(b.handle, s)
            ev[1].record(stream)
            for _ in range(steps):
                ihist.ihist_batch_query_all(b.handle, d_rects.data_ptr(), NRECTS, q.data_ptr(), s)
            ev[2].record(stream)
            torch.cuda.synchronize()
            if b.status() != ihist.IHIST_OK:
                raise SystemExit("device status error in the %s run" % name)
            scan_ms, query_ms = ev[0].elapsed_time(ev[1]) / steps, ev[1].elapsed_time(ev[2]) / steps
            out[name] = {"scan_ms": scan_ms, "query_ms": query_ms,
                         "frames_per_s": n * 1e3 / (scan_ms + query_ms), "scan_gbs": byts / scan_ms / 1e6}
        del q
    return out


def other_bins_report(d_frames, outs, stream, steps: int = 5) -> dict:
    """Per-frame launches with other bin structures on the same 1080p
    frames and output buffers: 64 non-uniform bins given by edges, and the
    joint 4 x 4 x 4 bins of three-channel frames.  Algorithmic bytes are the
    output words plus one read of the frame (three bytes per pixel for the
    joint case)."""
    import torch

    from paper_1711_01919_gb300 import ihist
    n = d_frames.shape[0]
    s = stream.cuda_stream
    edges = [3 * k + (k * k) // 64 for k in range(NBINS + 1)]  # widths 3..5, non-uniform
    rgb = torch.stack([d_frames, d_frames.roll(1, 0), d_frames.roll(2, 0)], dim=3).contiguous()
    out = {}
    for name, plan, inp, pitch, read_bytes in (
            ("edges_64_nonuniform", ihist.Plan(H, W, edges=edges), d_frames, W, H * W),
            ("joint_rgb_4x4x4", ihist.Plan(H, W, bins_per_channel=[4, 4, 4]), rgb, 3 * W, 3 * H * W)):

        def loop():
            for f in range(n):
                ihist.ihist_compute(plan.handle, inp[f].data_ptr(), pitch, outs[f].data_ptr(), s)

        for _ in range(3):
            loop()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record(stream)
        for _ in range(steps):
            loop()
        b.record(stream)
        torch.cuda.synchronize()
        if plan.status() != ihist.IHIST_OK:
            raise SystemExit("device status error in the %s run" % name)
        sec = a.elapsed_time(b) / 1000.0
        byts = steps * n * (H * W * NBINS * 4 + read_bytes)
        out[name] = {"frames_per_s": steps * n / sec, "gbs": byts / sec / 1e9,
                     "form": "%d x ihist_compute per step" % n, "tile": tile_of(plan)}
        plan.close()
    # the same frames in one batched launch each: the edges as value -> bin
    # tables, and the joint RGB bins (joint-bin planes, then one scan launch)
    for name, frames_in, kw, read_bytes in (
            ("edges_64_nonuniform_batched", [d_frames[f] for f in range(n)],
             {"tables": [ihist.edges_table(edges)] * n}, H * W),
            ("joint_rgb_4x4x4_batched", [rgb[f] for f in range(n)], {"joint": [[4, 4, 4]] * n}, 3 * H * W)):
        batch = ihist.Batch(frames_in, NBINS, outs=[outs[f] for f in range(n)], **kw)
        for _ in range(3):
            batch.compute(stream)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record(stream)
        for _ in range(steps):
            batch.compute(stream)
        b.record(stream)
        torch.cuda.synchronize()
        if batch.status() != ihist.IHIST_OK:
            raise SystemExit("device status error in the %s run" % name)
        sec = a.elapsed_time(b) / 1000.0
        byts = steps * n * (H * W * NBINS * 4 + read_bytes)
        out[name] = {"frames_per_s": steps * n / sec, "gbs": byts / sec / 1e9,
                     "form": "ihist_batch_compute over %d frames per step (%s)" % (n, ", ".join(kw)),
                     "tune": batch.tune}
        batch.close()
    del rgb
    return out


def main():
    global NFRAMES
    args = parse_args()
    if args.frames != NFRAMES:
        if args.frames < 2 or args.frames % 2:
            raise SystemExit("--frames must be an even number >= 2")
        NFRAMES = args.frames
    if args.impl == "reference":
        return run_reference(args)
    if args.case == "mp64-slice":
        return run_mp64_slice(args)
    if args.case == "query-slice":
        return run_query_slice(args)
    if args.case == "vga":
        return run_vga(args)
    import torch
    import torch.distributed as dist

    from paper_1711_01919_gb300 import build as cuda_build
    from paper_1711_01919_gb300 import ihist

    rank, world, local_rank = dist_env()
    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA GPU")
    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    if world > 1:
        dist.init_process_group("nccl", device_id=dev)
    if rank == 0 or not os.path.exists(cuda_build.LIB):
        cuda_build.build()
    if world > 1:
        dist.barrier()
    ihist.load()

    frames = make_frames(rank)
    from paper_1711_01919_gb300 import synth as _synth
    input_hashes = [hex(_synth.fnv1a64_rows(f)) for f in frames]  # FNV-1a 64 of each generated frame
    rects = make_rects()
    d_frames = torch.from_numpy(frames).to(dev)
    # every frame queries the same rectangles: [frames][rects][4]
    d_rects = torch.from_numpy(np.ascontiguousarray(np.broadcast_to(rects, (NFRAMES,) + rects.shape))).to(dev)
    layout = {"bin": ihist.IHIST_BIN_MAJOR, "pixel": ihist.IHIST_PIXEL_MAJOR,
              "quad": ihist.IHIST_QUAD_MAJOR}[args.layout]
    outs = torch.empty((NFRAMES,) + ihist.out_shape(H, W, NBINS, layout), dtype=torch.int32, device=dev)
    d_query = torch.empty((NFRAMES * NRECTS * NBINS,), dtype=torch.int32, device=dev)
    stream = torch.cuda.current_stream(dev)
    s = stream.cuda_stream

    # the batched form: one persistent launch over all 64 resident frames,
    # one launch for all 64 x 1000 region queries
    batch = ihist.Batch([d_frames[f] for f in range(NFRAMES)], NBINS, [layout] * NFRAMES,
                        outs=[outs[f] for f in range(NFRAMES)])
    rp, qp = d_rects.data_ptr(), d_query.data_ptr()

    def step():
        ihist.ihist_batch_compute(batch.handle, s)
        ihist.ihist_batch_query_all(batch.handle, rp, NRECTS, qp, s)

    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()
    if batch.status() != ihist.IHIST_OK:
        raise SystemExit("device status error during warm-up")

    # ---- device-resident timed region ----
    kev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    t_start, t_end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    clocks = ClockSampler(nvml_bus_id(dev))
    clocks.start()
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    t_start.record(stream)
    for k in range(args.steps):
        kev[k][0].record(stream)
        ihist.ihist_batch_compute(batch.handle, s)
        kev[k][1].record(stream)
        ihist.ihist_batch_query_all(batch.handle, rp, NRECTS, qp, s)
    t_end.record(stream)
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    try:
        props = torch.cuda.get_device_properties(dev)
        bus = "%02x:%02x.0" % (props.pci_bus_id, props.pci_device_id)
    except AttributeError:
        bus = None
    clk = clocks.stop(bus)
    elapsed_ms = t_start.elapsed_time(t_end)
    kernel_ms = [a.elapsed_time(b) for a, b in kev]
    if batch.status() != ihist.IHIST_OK:
        raise SystemExit("device status error during the timed region")
    resident_query = d_query.view(NFRAMES, NRECTS, NBINS)[NFRAMES - 1].cpu()

    # ---- plain per-frame launches (same frames, same outputs); then the
    # same with overlapped launches (no kernel in the step writes a frame) ----
    pf_steps = max(3, min(args.steps, 20))

    def time_plain(plan):
        def plain_step():
            for f in range(NFRAMES):
                ihist.ihist_compute(plan.handle, d_frames[f].data_ptr(), W, outs[f].data_ptr(), s)
                ihist.ihist_query(plan.handle, outs[f].data_ptr(), rp, NRECTS,
                                  d_query[f * NRECTS * NBINS:].data_ptr(), s)

        d_query.fill_(-1)
        for _ in range(2):
            plain_step()
        p_start, p_end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        p_start.record(stream)
        for _ in range(pf_steps):
            plain_step()
        p_end.record(stream)
        torch.cuda.synchronize()
        if plan.status() != ihist.IHIST_OK:
            raise SystemExit("device status error in the per-frame run")
        if not torch.equal(d_query.view(NFRAMES, NRECTS, NBINS)[NFRAMES - 1].cpu(), resident_query):
            raise SystemExit("per-frame and batched query results differ")
        return p_start.elapsed_time(p_end)

    plan = ihist.Plan(H, W, NBINS, layout)
    plain_ms = time_plain(plan)
    plan_ov = ihist.Plan(H, W, NBINS, layout, tune={"overlap": 1})
    overlap_ms = time_plain(plan_ov)

    # ---- end-to-end: pinned host frames -> copy stream -> batched compute ->
    # batched query -> host; two 32-frame batches alternate so one batch's
    # upload overlaps the other's compute, and the step's query rows go back
    # on a third stream under the next step's first compute ----
    e2e_steps = args.e2e_steps or min(args.steps, 30)
    half = NFRAMES // 2
    h_frames = torch.from_numpy(frames).pin_memory()
    h_query = torch.empty((NFRAMES * NRECTS * NBINS,), dtype=torch.int32).pin_memory()
    d_in2 = torch.empty((NFRAMES, H, W), dtype=torch.uint8, device=dev)
    halves = [ihist.Batch([d_in2[f] for f in range(g * half, (g + 1) * half)], NBINS, [layout] * half,
                          outs=[outs[f] for f in range(g * half, (g + 1) * half)]) for g in range(2)]
    copy_stream = torch.cuda.Stream(dev)
    d2h_stream = torch.cuda.Stream(dev)
    ev_queried, ev_copied = torch.cuda.Event(), torch.cuda.Event()
    ev_copied.record(d2h_stream)
    hq = [h_frames[f] for f in range(NFRAMES)]
    qsz = half * NRECTS * NBINS

    def e2e_step():
        for g in range(2):
            ihist.ihist_batch_upload_compute(halves[g].handle, [x.data_ptr() for x in hq[g * half:(g + 1) * half]],
                                             s, copy_stream.cuda_stream)
            if g == 0:
                stream.wait_event(ev_copied)  # the previous step's rows have left d_query
            ihist.ihist_batch_query_all(halves[g].handle, d_rects[g * half:].data_ptr(), NRECTS,
                                        d_query[g * qsz:].data_ptr(), s)
        ev_queried.record(stream)
        d2h_stream.wait_event(ev_queried)
        with torch.cuda.stream(d2h_stream):
            h_query.copy_(d_query, non_blocking=True)
        ev_copied.record(d2h_stream)

    for _ in range(2):
        e2e_step()
    torch.cuda.synchronize()
    e_start, e_end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    e_start.record(stream)
    copy_stream.wait_event(e_start)
    for _ in range(e2e_steps):
        e2e_step()
    stream.wait_event(ev_copied)  # the last step's result is on the host
    e_end.record(stream)
    torch.cuda.synchronize()
    e2e_ms = e_start.elapsed_time(e_end)
    for hb in halves:
        if hb.status() != ihist.IHIST_OK:
            raise SystemExit("device status error during the e2e region")
    if not torch.equal(h_query.view(NFRAMES, NRECTS, NBINS)[NFRAMES - 1], resident_query):
        raise SystemExit("e2e query results differ from the device-resident run")

    # ---- the per-frame form of the same pipeline (Algorithm 6): host frames
    # through a 2-slot device ring on the copy stream, one overlapped scan and
    # one query per frame, the query rows back to pinned host memory ----
    seq_plan = ihist.Plan(H, W, NBINS, layout)
    slots = torch.empty((2, H, W), dtype=torch.uint8, device=dev)
    d_q1 = torch.empty((NRECTS * NBINS,), dtype=torch.int32, device=dev)
    seq_steps = max(3, min(args.steps, 10))

    def seq_step():
        ihist.ihist_sequence_host(seq_plan.handle, h_frames.data_ptr(), H * W, NFRAMES, slots.data_ptr(),
                                  outs.data_ptr(), NFRAMES, d_rects.data_ptr(), NRECTS, d_q1.data_ptr(),
                                  h_query.data_ptr(), s, copy_stream.cuda_stream)

    for _ in range(2):
        seq_step()
    torch.cuda.synchronize()
    q_start, q_end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    q_start.record(stream)
    copy_stream.wait_event(q_start)
    for _ in range(seq_steps):
        seq_step()
    q_end.record(stream)
    torch.cuda.synchronize()
    seq_ms = q_start.elapsed_time(q_end)
    if seq_plan.status() != ihist.IHIST_OK:
        raise SystemExit("device status error in the per-frame sequence")
    if not torch.equal(h_query.view(NFRAMES, NRECTS, NBINS)[NFRAMES - 1], resident_query):
        raise SystemExit("per-frame sequence query results differ from the batched run")
    seq_plan.close()
    del slots, d_q1

    other_bins = None if args.no_configs else other_bins_report(d_frames, outs, stream)
    layouts = None if args.no_configs else layouts_report(d_frames, outs, d_rects, stream)

    # ---- write-only probe: the store bandwidth a plain fill reaches on this GPU ----
    probe = torch.empty((1 << 30,), dtype=torch.int32, device=dev)
    for _ in range(3):
        probe.fill_(1)
    w_start, w_end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    w_start.record(stream)
    for _ in range(10):
        probe.fill_(1)
    w_end.record(stream)
    torch.cuda.synchronize()
    write_probe_gbs = 10 * probe.numel() * 4 / (w_start.elapsed_time(w_end) / 1000.0) / 1e9
    del probe

    elapsed_ms, e2e_ms, plain_ms, overlap_ms, seq_ms = max_over_ranks(
        [elapsed_ms, e2e_ms, plain_ms, overlap_ms, seq_ms], world, dev)

    if rank == 0:
        value = job_throughput(NFRAMES, args.steps, world, elapsed_ms)
        peak, peak_kind = measured_peak()
        bytes_per_launch = NFRAMES * algorithmic_bytes_per_frame()
        mean_kernel_s = statistics.fmean(kernel_ms) / 1000.0
        achieved = bytes_per_launch / mean_kernel_s / 1e9
        line = {
            "metric": METRIC, "value": value, "unit": "frames/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": elapsed_ms / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "u32", "data": "synthetic",
            "config": {
                "workload": WORKLOAD, "frames_per_step": NFRAMES, "H": H, "W": W, "B": NBINS,
                "layout": {ihist.IHIST_BIN_MAJOR: "bin-major", ihist.IHIST_PIXEL_MAJOR: "pixel-major",
                           ihist.IHIST_QUAD_MAJOR: "quad-major"}[layout],
                "queries_per_frame": NRECTS,
                "input_fnv1a64": input_hashes,
                "form": "batched: one persistent scan launch over the %d resident frames + one query launch" % NFRAMES,
                "parallelism": "replicas (one independent 64-frame sequence per GPU)" if world > 1 else "single GPU",
                "l2": "no flush: each step writes %.1f GB of output, > 129 MB L2" % (NFRAMES * H * W * NBINS * 4 / 1e9),
                "written_gbs": world * NFRAMES * args.steps * H * W * NBINS * 4 / (elapsed_ms / 1000.0) / 1e9,
                "batch_items_per_launch": batch.items(),
                "scan_launch_ms_median": statistics.median(kernel_ms),
                "plain_per_frame": {
                    "value": job_throughput(NFRAMES, pf_steps, world, plain_ms), "unit": "frames/s",
                    "steps": pf_steps, "form": "%d x (ihist_compute + ihist_query) per step" % NFRAMES,
                    "tile": tile_of(plan)},
                "plain_per_frame_overlapped": {
                    "value": job_throughput(NFRAMES, pf_steps, world, overlap_ms), "unit": "frames/s",
                    "steps": pf_steps, "form": "as plain_per_frame, plan tune overlap=1 (programmatic "
                                               "dependent launch: each scan starts while the kernel before it "
                                               "finishes)"},
            },
            "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                         "frac": achieved / peak, "traffic": profiled_traffic(),
                         "kernel": "ihist::batch_kernel (%d frames per launch)" % NFRAMES,
                         "bytes_per_launch": bytes_per_launch,
                         "peak_source": "%s (MEASURED_PEAKS.json hbm_gbs)" % peak_kind,
                         "write_probe_gbs": write_probe_gbs,
                         "frac_of_write_probe": achieved / write_probe_gbs},
            "e2e": {"value": job_throughput(NFRAMES, e2e_steps, world, e2e_ms), "unit": "frames/s",
                    "h2d_bytes_per_step": NFRAMES * H * W, "d2h_bytes_per_step": NFRAMES * NRECTS * NBINS * 4,
                    "steps": e2e_steps,
                    "api": "ihist_batch_upload_compute on two alternating %d-frame batches (pinned host frames, "
                           % (NFRAMES // 2) +
                           "copy stream) + ihist_batch_query_all + copy of the query results to pinned host "
                           "(on a third stream, under the next step's first compute)",
                    "per_frame_sequence": {
                        "value": job_throughput(NFRAMES, seq_steps, world, seq_ms), "unit": "frames/s",
                        "steps": seq_steps,
                        "api": "ihist_sequence_host: pinned host frames through a 2-slot device ring on the copy "
                               "stream, one scan (overlapped launch) + one ihist_query per frame, each frame's "
                               "query rows back to pinned host"}},
            "gpu_launches": 2 * args.steps,
            "clocks": clk,
        }
        if not args.no_configs:
            for v in other_bins.values():
                v["frac"] = v["gbs"] / peak
            line["other_bins"] = other_bins
            for v in layouts.values():
                v["scan_frac"] = v["scan_gbs"] / peak
            line["layouts_64x1080p_b64_1000q"] = layouts
            line["other_workloads"] = configs_report(stream, peak)
        if args.serve_seconds > 0:
            line["serving"] = serving_report(args.serve_seconds)
        if not args.no_cpu_baseline:
            import oracle
            oracle.build()
            line["cpu_baseline"] = cpu_baseline(frames, args.cpu_seconds, 1)
            line["cpu_baseline_all_cores"] = cpu_baseline(frames, args.cpu_seconds / 2, host_cores())
        print(json.dumps(line), flush=True)
    for hb in halves:
        hb.close()
    batch.close()
    plan.close()
    if world > 1:
        dist.barrier()
        dist.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
