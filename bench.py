#!/usr/bin/env python
"""Benchmark of the single-pulse search: searched DM x time samples per second.

Workload (default): the SKA-like FP32 chunk -- 4096 DM trials x 524288 samples
(33.5 s at 64 us), N(100, 12^2) noise with a +-2 sigma sinusoidal baseline
drift of period 2^16 samples, 200 Gaussian pulses; widths 1..16 then 24..256
in steps of 8 (46 widths); threshold 7; sigma_N = sqrt(N) sigma; one MSD for
the whole plane.  A step is one whole search (MSD partial + merge kernels,
then the fused boxcar / SNR / max / threshold kernel) over the plane resident
in HBM, including the read-back of the candidate count.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl spd|reference]

Prints ONE JSON line (rank 0).  Under torchrun every rank searches its own
plane (independent chunks, weak scaling, no collective on the data path).
"""
from __future__ import annotations

import argparse
import ctypes
import hashlib
import json
import math
import os
import select
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "DM×time samples/s searched and real-time factor at SKA-like size; % HBM peak"
UNIT = "DM×time samples/s"
WIDTHS = list(range(1, 17)) + list(range(24, 257, 8))
THRESHOLD = 7.0
SAMPLE_TIME_S = 64e-6
# msd_partial, msd_merge_l1, fold_final, merge_shards, consts, screen, search
KERNELS_PER_STEP = 7
PROFILES = os.path.join(ROOT, "profiles")
# the kernels of the detect phase: the screen and the search of what it keeps
DETECT_SRC = [os.path.join(ROOT, "paper_1611_09704_gb300", "csrc", f)
              for f in ("spd_search_kernel.cuh", "spd_live.cuh", "spd_screen.cu")]


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["spd", "reference"], default="spd")
    ap.add_argument("--n-dm", type=int, default=4096)
    ap.add_argument("--n-samp", type=int, default=524288)
    ap.add_argument("--e2e-steps", type=int, default=8)
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--cpu-rows", type=int, default=1024)
    ap.add_argument("--ref-budget-s", type=float, default=150.0)
    ap.add_argument("--workload", choices=["ska", "plain", "precision", "batched", "serving",
                                           "decimated", "cluster", "plane", "dedisperse"],
                    default="ska",
                    help="ska: the SKA-like FP32 chunk (default, the headline); plain: 64 x 65536 "
                         "FP32 noise + top-hats; precision: the SKA-like chunk stored as FP16 / "
                         "BF16 with Eq. 5; batched: four decimated DM ranges in one launch; "
                         "serving: 16 beams of FP16 chunks streamed with continuous batching; "
                         "decimated: widths to 512 by decimation in time vs the plain search; "
                         "cluster: per-DM clustering of the SKA-like chunk's candidates; "
                         "plane: the unfused calls on the SKA-like chunk (spd_boxcar_snr, "
                         "spd_threshold_candidates); dedisperse: the de-dispersion producer")
    ap.add_argument("--beams", type=int, default=16)
    ap.add_argument("--chunks-per-beam", type=int, default=3)
    ap.add_argument("--slots", type=int, default=4)
    ap.add_argument("--compress", type=float, default=8.0,
                    help="serving: data time / wall time of the arrival schedule")
    ap.add_argument("--mem-budget-gb", type=float, default=32.0)
    ap.add_argument("--dtype", choices=["f16", "bf16"], default="f16")
    return ap.parse_args()


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            p = json.load(f)
        return float(p["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


def detect_source_sha() -> str:
    h = hashlib.sha256()
    for path in DETECT_SRC:
        with open(path, "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:16]


def traffic_file(workload: str) -> str:
    return os.path.join(PROFILES, f"traffic_search_{workload}.txt")


def _recorded(workload: str = "ska_like"):
    """The committed ncu record of one search-kernel launch on `workload`, or
    None when absent or taken on a different kernel source."""
    try:
        kv = {}
        with open(traffic_file(workload)) as f:
            for line in f:
                if ":" in line and not line.startswith("#"):
                    k, v = line.split(":", 1)
                    kv[k.strip()] = v.strip()
        return kv if kv.get("kernel_source_sha256") == detect_source_sha() else None
    except OSError:
        return None


def recorded_traffic(n_samples: int, n_cand: int, workload: str = "ska_like"):
    """DRAM bytes per search launch from the committed ncu record, scaled to
    this launch (reads by samples, writes by candidates); None without one."""
    kv = _recorded(workload)
    if kv is None:
        return None
    read = float(kv["dram_read_bytes"]) * n_samples / float(kv["samples"])
    write = float(kv["dram_write_bytes"]) * max(n_cand, 1) / max(float(kv["candidates"]), 1)
    return int(read + write)


def recorded_instructions(n_samples: int, workload: str = "ska_like"):
    """Issued warp instructions per search launch from the committed ncu
    record, scaled by samples (same data recipe); None without one."""
    kv = _recorded(workload)
    if kv is None or "warp_instructions" not in kv:
        return None
    return float(kv["warp_instructions"]) * n_samples / float(kv["samples"])


def hbm_roofline(kernel: str, alg_bytes: float, ms: float, traffic=None, note=None):
    """Roofline object of one kernel (or step) bound by HBM: algorithmic bytes
    over the CUDA-event time, against the measured copy bandwidth."""
    hbm, kind = peaks()
    ach = alg_bytes / (ms / 1e3) / 1e9
    r = {"bound": "hbm", "kernel": kernel, "achieved": ach, "peak": hbm, "unit": "GB/s",
         "frac": ach / hbm, "traffic": traffic, "peak_source": f"{kind} hbm_gbs",
         "algorithmic_bytes": int(alg_bytes), "ms": ms}
    if note:
        r["note"] = note
    return r


def sm_max_mhz() -> float:
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return float(json.load(f).get("sm_max_mhz") or 2070.0)
    except (OSError, ValueError):
        return 2070.0


def alu_roofline(kernel: str, ops: float, ms: float, note=None):
    """Roofline object of a kernel bound by FP32 arithmetic: algorithmic
    operations over the CUDA-event time, against SMs x 128 FP32 lanes x 2
    (packed f32x2 add / multiply) x the measured maximum SM clock."""
    mhz = sm_max_mhz()
    peak = SM_COUNT * 128 * 2 * mhz * 1e6 / 1e12
    ach = ops / (ms / 1e3) / 1e12
    r = {"bound": "alu", "kernel": kernel, "achieved": ach, "peak": peak, "unit": "Tops/s",
         "frac": ach / peak, "traffic": None,
         "peak_source": f"{SM_COUNT} SMs x 128 lanes x 2 (f32x2) x {mhz:.0f} MHz",
         "algorithmic_ops": ops, "ms": ms}
    if note:
        r["note"] = note
    return r


def lds_roofline(kernel: str, words: float, ms: float, note=None):
    """Roofline object of a kernel bound by shared-memory reads (one 32-bit
    word per arithmetic operation): words over the CUDA-event time, against
    SMs x 32 words per clock x the measured maximum SM clock."""
    mhz = sm_max_mhz()
    peak = SM_COUNT * 32 * mhz * 1e6 / 1e12
    ach = words / (ms / 1e3) / 1e12
    r = {"bound": "alu", "kernel": kernel, "achieved": ach, "peak": peak, "unit": "Twords/s",
         "frac": ach / peak, "traffic": None,
         "peak_source": f"{SM_COUNT} SMs x 32 shared-memory words/clk x {mhz:.0f} MHz",
         "algorithmic_words": words, "ms": ms}
    if note:
        r["note"] = note
    return r


SM_COUNT, SCHEDULERS_PER_SM = 152, 4


class Clocks:
    """nvidia-smi sampling of SM clock and throttle reasons during the timed region."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device_index):
        self.p = None
        self.lines = []
        try:
            import torch
            uuid = str(torch.cuda.get_device_properties(device_index).uuid)
            sel = uuid if uuid.startswith("GPU-") else "GPU-" + uuid
            self.p = subprocess.Popen(
                ["nvidia-smi", "-i", sel, f"--query-gpu={self.Q}", "--format=csv,noheader,nounits",
                 "-lms", "100"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            # nvidia-smi's start-up (NVML initialisation) slows the CUDA calls of
            # this process for a while: wait for its first sample, which is then
            # dropped, so that the timed region begins after it
            if select.select([self.p.stdout], [], [], 10.0)[0]:
                self.p.stdout.readline()
        except Exception:
            self.p = None

    def stop(self):
        if self.p is None:
            return None
        time.sleep(0.15)
        self.p.terminate()
        try:
            out, _ = self.p.communicate(timeout=5)
        except Exception:
            self.p.kill()
            out = ""
        return self.parse(out)

    @staticmethod
    def parse(out: str):
        """Summary of nvidia-smi CSV samples (the Q fields, no units): median SM
        clock, highest maximum clock, and the throttle reasons seen active."""
        sm, mx, reasons = [], 0.0, set()
        for line in out.strip().splitlines():
            f = [x.strip() for x in line.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx = max(mx, float(f[2]))
            except ValueError:
                continue
            for name, v in zip(["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown",
                                "sw_power_cap"], f[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(name)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": mx, "reasons": sorted(reasons),
                "samples": len(sm)}


def issue_roofline(n_samples: int, det_ms: float):
    """The bound the detect kernel actually meets: instruction issue.  achieved
    = recorded warp instructions (ncu, scaled to this launch) / the live
    CUDA-event time; peak = one warp instruction per scheduler per cycle at the
    measured maximum SM clock."""
    inst = recorded_instructions(n_samples)
    mhz = None
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            mhz = json.load(f).get("sm_max_mhz")
    except (OSError, ValueError):
        pass
    mhz = mhz or 2070.0
    peak = SM_COUNT * SCHEDULERS_PER_SM * mhz * 1e6 / 1e12      # T warp-instr/s
    if inst is None:
        return {"bound": "issue", "achieved": None, "peak": peak, "unit": "Twarp-inst/s",
                "frac": None, "note": "no ncu record for this kernel source"}
    ach = inst / (det_ms / 1e3) / 1e12
    return {"bound": "issue", "achieved": ach, "peak": peak, "unit": "Twarp-inst/s",
            "frac": ach / peak, "warp_instructions": inst,
            "peak_source": f"{SM_COUNT} SMs x {SCHEDULERS_PER_SM} schedulers x {mhz:.0f} MHz"}


def workload_config(n_dm, n_samp, world):
    return {"workload": (f"SKA-like FP32 chunk {n_dm} DM x {n_samp} samples (64 us), "
                         "N(100,12^2) + 2-sigma drift + 200 Gaussian pulses; widths 1..16 + "
                         "24..256/8 (46); f_T 7; sqrt(N) sigma; global MSD"),
            "n_dm": n_dm, "n_samp": n_samp, "n_widths": len(WIDTHS), "threshold": THRESHOLD,
            "dtype_in": "f32", "l2": "inputs larger than L2 (plane %.2f GB)" % (n_dm * n_samp * 4 / 1e9),
            "parallelism": (f"DM-row shards x{world}: {n_dm} rows per GPU, one MSD over all "
                            f"{n_dm * world} rows (all-gather of 40-byte Chan partials)"
                            if world > 1 else "one GPU")}


# ------------------------------------------------------------------ CPU side

def oracle_sample(rows, n_samp, seed):
    """The oracle (FP64, OpenMP over rows) on `rows` rows of the SKA-like recipe."""
    import oracle
    import synth
    sp = synth.ska_like(rows, n_samp, n_pulses=max(1, 200 * rows // 4096), device="cpu",
                        seed=seed)
    x = synth.to_host_numpy(sp.data)
    oracle.build()
    t0 = time.perf_counter()
    cands, _, _, _ = oracle.search(x, WIDTHS, THRESHOLD)
    dt = time.perf_counter() - t0
    return dt, cands.size, oracle.num_threads()


def run_reference(a, rank, world):
    if rank != 0:
        return 0
    n_samp = a.n_samp
    # calibrate the per-row cost, then size each step to fit the time budget
    dt16, _, cores = oracle_sample(16, n_samp, 5)
    per_row = dt16 / 16
    rows = int(max(8, min(512, a.ref_budget_s / max(1, a.steps + a.warmup) / per_row)))
    for w in range(a.warmup):
        oracle_sample(rows, n_samp, 100 + w)
    times = []
    for k in range(a.steps):
        dt, _, cores = oracle_sample(rows, n_samp, 1000 + k)
        times.append(dt)
    t = sum(times) / len(times)
    value = rows * n_samp / t
    line = {"metric": METRIC, "value": value, "unit": UNIT, "impl": "reference",
            "n_gpus": world, "steps": a.steps, "warmup": a.warmup, "ms_per_step": t * 1e3,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": workload_config(a.n_dm, n_samp, 1),
            "realtime_factor": n_samp * SAMPLE_TIME_S / (t * a.n_dm / rows),
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle",
                             "sample": f"{rows} rows x {n_samp} samples per step "
                                       "(same recipe), MSD over the sample"},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}
    print(json.dumps(line))
    return 0


# ------------------------------------------------------------------ GPU side

def run_spd(a, rank, world, local):
    import torch
    import torch.distributed as dist

    import paper_1611_09704_gb300 as spd
    import synth
    from paper_1611_09704_gb300.sharding import ShardedSearch

    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    spd.build()
    spd.load()
    n_dm, n_samp = a.n_dm, a.n_samp
    n = n_dm * n_samp
    sp = synth.ska_like(n_dm, n_samp, device=dev, seed=1611_1 + rank)
    x = sp.data
    cap = int(n * 0.45) + 1024
    # this rank's DM rows [rank * n_dm, (rank + 1) * n_dm) of the whole plane
    ss = ShardedSearch(x, WIDTHS, THRESHOLD, cap, dm_offset=rank * n_dm)
    res = ss.result
    res_host = torch.empty(16, dtype=torch.uint8, pin_memory=True)
    stream = torch.cuda.current_stream()

    def step(e0=None, e1=None, e2=None):
        if e0 is not None:
            e0.record(stream)
        ss.msd_step()          # shard partial, all-gather (N > 1), Eq. 2 merge
        if e1 is not None:
            e1.record(stream)
        ss.detect_step()       # fused boxcar + SNR + max + threshold
        if e2 is not None:
            e2.record(stream)
        res_host.copy_(res, non_blocking=True)

    for _ in range(max(3, a.warmup)):
        step()
    torch.cuda.synchronize()
    count, status = spd.read_result(res)
    if status != 0:
        raise RuntimeError(f"search status {status}")
    if count > cap:
        raise RuntimeError(f"{count} candidates exceed capacity {cap}")

    ev = [[torch.cuda.Event(enable_timing=True) for _ in range(3)] for _ in range(a.steps)]
    t_start = torch.cuda.Event(enable_timing=True)
    t_end = torch.cuda.Event(enable_timing=True)
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    clk = Clocks(local) if rank == 0 else None
    t_start.record(stream)
    for k in range(a.steps):
        step(*ev[k])
    t_end.record(stream)
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    clocks = clk.stop() if clk else None
    total_ms = t_start.elapsed_time(t_end)
    msd_ms = statistics.mean(e[0].elapsed_time(e[1]) for e in ev)
    det_ms = statistics.mean(e[1].elapsed_time(e[2]) for e in ev)
    if world > 1:
        t = torch.tensor([total_ms], device=dev)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        total_ms = float(t.item())
    ms_step = total_ms / a.steps
    value = world * n / (ms_step / 1e3)
    e2e_line = None
    if not a.no_e2e:
        e2e_line = e2e(x, count, a.e2e_steps, n, world, rank, dev)
        link = host_link(dev)
        hb, db = e2e_line["h2d_bytes_per_step"], e2e_line["d2h_bytes_per_step"]
        # lower bound of a plane's time from the link alone: neither direction
        # faster than alone, both together no faster than the duplex aggregate
        link["bound_ms_per_step"] = 1e3 * max(
            hb / (link["h2d_gbs"] * 1e9), db / (link["d2h_gbs"] * 1e9),
            (hb + db) / (2 * link["duplex_gbs_each"] * 1e9))
        e2e_line["host_link"] = link
    if rank != 0:
        return 0

    hbm, peak_kind = peaks()
    det_bytes = n * 4 + 16 * count
    traffic = recorded_traffic(n, count)
    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": a.steps,
            "warmup": a.warmup, "ms_per_step": ms_step, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": workload_config(n_dm, n_samp, world),
            "realtime_factor": n_samp * SAMPLE_TIME_S / (ms_step / 1e3),
            "candidates_per_step": count,
            "roofline": hbm_roofline("screen_kernel + search_kernel (boxcar + SNR + max + threshold)",
                                     det_bytes, det_ms, traffic),
            "issue_roofline": issue_roofline(n, det_ms),
            "step_breakdown_ms": {"msd": msd_ms, "detect": det_ms},
            "whole_step_hbm_frac": (2 * n * 4 + 16 * count) / (ms_step / 1e3) / 1e9 / hbm,
            "gpu_launches": KERNELS_PER_STEP * a.steps,
            "clocks": clocks}

    if not a.no_e2e:
        line["e2e"] = e2e_line
    if not a.no_cpu_baseline:
        rows = min(a.cpu_rows, n_dm)
        dt, _, cores = oracle_sample(rows, n_samp, 7)
        line["cpu_baseline"] = {"value": rows * n_samp / dt, "unit": UNIT, "cores": cores,
                                "kind": "oracle",
                                "sample": f"{rows} rows x {n_samp} samples of the same recipe, "
                                          f"oracle MSD over the sample, {dt:.1f} s"}
    print(json.dumps(line))
    return 0


def host_link(dev, nbytes=1 << 30, reps=3):
    """Page-locked host <-> device copy rates (GB/s) of this GPU's host link:
    each direction alone and both at once on two streams, CUDA-event timed."""
    import torch
    h = torch.empty(nbytes, dtype=torch.uint8, pin_memory=True)
    h2 = torch.empty(nbytes, dtype=torch.uint8, pin_memory=True)
    d = torch.empty(nbytes, dtype=torch.uint8, device=dev)
    d2 = torch.empty(nbytes, dtype=torch.uint8, device=dev)
    s1, s2 = torch.cuda.Stream(device=dev), torch.cuda.Stream(device=dev)

    def rate(fn):
        fn()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for _ in range(reps):
            fn()
        torch.cuda.synchronize()
        return reps * nbytes / (time.perf_counter() - t0) / 1e9

    def h2d():
        with torch.cuda.stream(s1):
            d.copy_(h, non_blocking=True)

    def d2h():
        with torch.cuda.stream(s2):
            h2.copy_(d2, non_blocking=True)

    def both():
        h2d()
        d2h()

    # both(): nbytes each way per repetition, so its rate is per direction
    r = {"h2d_gbs": rate(h2d), "d2h_gbs": rate(d2h), "duplex_gbs_each": rate(both)}
    del h, h2, d, d2
    torch.cuda.empty_cache()
    return r


def e2e(x, count, steps, n, world, rank, dev):
    """Planes searched from page-locked host memory through spd_search_host,
    the C-ABI call with host buffers: every call copies its plane in, computes
    the MSD and searches, and returns with every candidate record and the
    count in host memory.  Two host threads call it with their own stream and
    workspace, so one plane's copy in overlaps the other's copy out.
    Whole-run wall time / planes, slowest rank (each rank's plane its own
    dataset: MSD per plane)."""
    import threading

    import torch
    import torch.distributed as dist

    import paper_1611_09704_gb300 as spd
    local = dev.index if dev.index is not None else 0
    xh = torch.empty(x.shape, dtype=x.dtype, pin_memory=True)
    xh.copy_(x)
    cap = count + (count >> 4) + 1024
    n_workers = 2
    ws = [torch.empty(spd.search_host_workspace_bytes(xh, WIDTHS, THRESHOLD, cap),
                      dtype=torch.uint8, device=dev) for _ in range(n_workers)]
    outs = [torch.empty((cap, 4), dtype=torch.int32, pin_memory=True) for _ in range(n_workers)]
    streams = [torch.cuda.Stream(device=dev) for _ in range(n_workers)]
    counts = [[] for _ in range(n_workers)]
    errors = []

    def worker(w, planes):
        try:
            torch.cuda.set_device(local)
            for _ in range(planes):
                c, st = spd.search_host(xh, WIDTHS, THRESHOLD, outs[w], workspace=ws[w],
                                        stream=streams[w])
                if st != 0 or c != count:
                    raise RuntimeError(f"spd_search_host: count {c} status {st}")
                counts[w].append(c)
        except Exception as e:   # reported by the caller
            errors.append(e)

    def run(planes):
        th = [threading.Thread(target=worker, args=(w, planes // n_workers + (w < planes % n_workers)))
              for w in range(n_workers)]
        for t in th:
            t.start()
        for t in th:
            t.join()
        if errors:
            raise errors[0]

    run(n_workers)          # untimed: set-up, page-in of the host buffers
    for c in counts:
        c.clear()
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    run(steps)
    t = (time.perf_counter() - t0) / steps
    if world > 1:
        tt = torch.tensor([t], device=dev)
        dist.all_reduce(tt, op=dist.ReduceOp.MAX)
        t = float(tt.item())
    del ws, outs
    torch.cuda.empty_cache()
    return {"value": world * n / t, "unit": UNIT, "h2d_bytes_per_step": n * x.element_size(),
            "d2h_bytes_per_step": 16 + 16 * count, "ms_per_step": t * 1e3, "steps": steps,
            "api": f"spd_search_host (C ABI, host buffers: page-locked plane in, records and "
                   f"count out) from {n_workers} host threads"}


def timed(step, steps, warmup, clocks_dev):
    """Warm up, then time `steps` calls of step() with CUDA events."""
    import torch
    for _ in range(max(3, warmup)):
        step()
    torch.cuda.synchronize()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    clk = Clocks(clocks_dev)
    e0.record()
    for _ in range(steps):
        step()
    e1.record()
    torch.cuda.synchronize()
    return e0.elapsed_time(e1) / steps, clk.stop()


def timed_split(phases, steps, warmup, clocks_dev):
    """Warm up, then time `steps` passes of the phases (callables run in
    order) with CUDA events between them on the current stream: returns
    (total ms per step, [ms per step of each phase], clocks)."""
    import torch
    for _ in range(max(3, warmup)):
        for f in phases:
            f()
    torch.cuda.synchronize()
    ev = [[torch.cuda.Event(enable_timing=True) for _ in range(len(phases) + 1)]
          for _ in range(steps)]
    clk = Clocks(clocks_dev)
    for k in range(steps):
        ev[k][0].record()
        for j, f in enumerate(phases):
            f()
            ev[k][j + 1].record()
    torch.cuda.synchronize()
    clocks = clk.stop()
    per = [statistics.mean(e[j].elapsed_time(e[j + 1]) for e in ev) for j in range(len(phases))]
    total = statistics.mean(e[0].elapsed_time(e[-1]) for e in ev)
    return total, per, clocks


def run_other(a):
    """The other configurations of the search, one JSON line each."""
    import torch

    import numpy as np

    import paper_1611_09704_gb300 as spd
    import synth

    local = int(os.environ.get("LOCAL_RANK", "0"))
    dev = torch.device("cuda", local)
    torch.cuda.set_device(local)
    spd.build()
    spd.load()
    hbm, peak_kind = peaks()
    line = {"metric": METRIC, "unit": UNIT, "n_gpus": 1, "steps": a.steps, "warmup": a.warmup,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "data": "synthetic", "workload_kind": a.workload}

    if a.workload == "plain":
        sp = synth.plain_tophat(64, 65536, device=dev, seed=1611_0)
        widths, thr = list(range(1, 33)), 6.0
        n = 64 * 65536
        out = torch.empty((1 << 20, 4), dtype=torch.int32, device=dev)
        res = torch.zeros(16, dtype=torch.uint8, device=dev)
        msd = torch.empty(40, dtype=torch.uint8, device=dev)
        ws = torch.empty(spd.search_workspace_bytes(sp.data, widths, thr), dtype=torch.uint8,
                         device=dev)
        step = lambda: spd.search(sp.data, widths, thr, out.shape[0], out=out, result=res,
                                  msd_out=msd, workspace=ws)
        ms, clocks = timed(step, a.steps, a.warmup, 0)
        count = spd.read_result(res)[0]
        line.update(value=n / (ms / 1e3), ms_per_step=ms, dtype="f32", clocks=clocks,
                    candidates_per_step=count, gpu_launches=4 * a.steps,
                    roofline=hbm_roofline("search step (MSD + search kernel)",
                                          2 * 4 * n + 16 * count, ms,
                                          note="inputs L2-resident (16.8 MB): latency-bound"),
                    realtime_factor=65536 * SAMPLE_TIME_S / (ms / 1e3),
                    config={"workload": "plain FP32 64 DM x 65536, N(0,1) + top-hats "
                                        "{1,3,8,17,30}; widths 1..32; f_T 6; sqrt(N) sigma",
                            "l2": "L2-resident (16.8 MB): latency-bound, no roofline"})
        print(json.dumps(line))
        return 0

    if a.workload == "precision":
        n_dm, n_samp = a.n_dm, a.n_samp
        sp, rows = synth.precision_plane(n_dm, n_samp, device=dev)
        q = synth.quantise_rows(sp, a.dtype)
        del sp
        torch.cuda.empty_cache()
        widths = WIDTHS
        x, scale = q.data, q.scale
        n = n_dm * n_samp
        out = torch.empty((int(n * 0.45) + 1024, 4), dtype=torch.int32, device=dev)
        res = torch.zeros(16, dtype=torch.uint8, device=dev)
        msd = torch.empty(40, dtype=torch.uint8, device=dev)
        modes = {}
        mws = torch.empty(max(spd.binding.load().spd_msd_workspace_bytes(
            ctypes.byref(spd.Plane(x, scale=scale).c()), 0, 256), 1), dtype=torch.uint8,
            device=dev)
        for mode, name in ((1, "eq5_as_printed"), (2, "eq5_linear_excess")):
            prm, keep = spd.binding._params(widths, THRESHOLD, mode, 0, 256)
            dws = torch.empty(spd.binding.load().spd_detect_workspace_bytes(
                ctypes.byref(spd.Plane(x, scale=scale).c()), ctypes.byref(prm)),
                dtype=torch.uint8, device=dev)
            del keep
            phases = [lambda: spd.msd(x, 0, 256, out=msd, workspace=mws, scale=scale),
                      lambda mode=mode: spd.detect(x, msd, widths, THRESHOLD, out.shape[0], mode,
                                                   0, 256, out=out, result=res, workspace=dws,
                                                   scale=scale)]
            ms, (msd_ms, det_ms), clocks = timed_split(phases, a.steps, a.warmup, 0)
            cnt = spd.read_result(res)[0]
            m = spd.msd_to_numpy(msd)[0]
            modes[name] = {"value": n / (ms / 1e3), "ms_per_step": ms, "candidates": cnt,
                           "step_breakdown_ms": {"msd_and_sigma_nmax": msd_ms, "detect": det_ms},
                           "mean": float(m["mean"]), "sd": float(m["sd"]),
                           "sd_nmax": float(m["sd_nmax"]), "clocks": clocks}
        main_ = modes["eq5_as_printed"]
        in_bytes = n * x.element_size()
        bd = main_["step_breakdown_ms"]
        line.update(value=main_["value"], ms_per_step=main_["ms_per_step"], dtype=a.dtype,
                    clocks=main_["clocks"], candidates_per_step=main_["candidates"],
                    gpu_launches=7 * a.steps, modes=modes,
                    roofline=hbm_roofline("screen_kernel + search_kernel (boxcar + SNR + max + threshold)",
                                          in_bytes + 16 * main_["candidates"], bd["detect"],
                                          recorded_traffic(n, main_["candidates"],
                                                           f"precision_{a.dtype}")),
                    msd_roofline=hbm_roofline("MSD (Eq. 1-2) and sigma_Nmax (Eq. 5) passes",
                                              2 * in_bytes, bd["msd_and_sigma_nmax"],
                                              note="two reads of the plane"),
                    error_vs_fp64_oracle="tests/test_gpu_precision_error.py (asserted bounds)",
                    realtime_factor=n_samp * SAMPLE_TIME_S / (main_["ms_per_step"] / 1e3),
                    whole_step_hbm_frac=(3 * in_bytes + 16 * main_["candidates"]) /
                    (main_["ms_per_step"] / 1e3) / 1e9 / hbm,
                    config={"workload": f"SKA-like chunk {n_dm} x {n_samp} stored as {a.dtype} "
                                        "with per-row scale; 5% rows with a 4000-sample pulse "
                                        "train (SNR 200); widths 1..16 + 24..256/8; f_T 7; Eq. 5 "
                                        "with sigma_Nmax at Nmax = 256",
                            "l2": "inputs larger than L2"})
        print(json.dumps(line))
        return 0

    if a.workload == "batched":
        from paper_1611_09704_gb300 import autotune
        specs, off, n, dur = [], 0, 0, 0.0
        planes = synth.batched_ranges(1.0, device=dev)
        for sp, dec, widths in planes:
            specs.append(spd.RangeSpec(sp.data, widths, THRESHOLD, dm_offset=off, decimation=dec))
            off += sp.n_dm
            n += sp.n_dm * sp.n_samp
            dur = sp.n_samp * dec * SAMPLE_TIME_S
        cap = 1 << 24
        tune = autotune.autotune(specs, cap, reps=3)
        bs = spd.BatchedSearch(specs, cap, tuning=tune["tuning"], graph=True)
        ms, clocks = timed(lambda: bs.run(), a.steps, a.warmup, 0)
        cnt = spd.read_result(bs.result)[0]
        in_bytes = n * 4
        line.update(value=n / (ms / 1e3), ms_per_step=ms, dtype="f32", clocks=clocks,
                    candidates_per_step=cnt, gpu_launches=(2 * len(specs) + 2) * a.steps,
                    tuning=tune, realtime_factor=dur / (ms / 1e3),
                    roofline=hbm_roofline("batched step (per-range MSD + one search-kernel "
                                          "launch), one graph replay", 2 * in_bytes + 16 * cnt,
                                          ms, note="the graph is timed whole: MSD reads each "
                                                   "range once more"),
                    whole_step_hbm_frac=(2 * in_bytes + 16 * cnt) / (ms / 1e3) / 1e9 / hbm,
                    config={"workload": "4 DM ranges, decimation 1/2/4/8: 2048x524288, "
                                        "1536x262144, 1024x131072, 512x65536 FP32 N(0,1) + "
                                        "Gaussian pulses; widths 1..64/128/256/512; f_T 7; "
                                        "one persistent launch in a CUDA graph",
                            "samples": n, "l2": "inputs larger than L2 (6.58 GB)"})
        print(json.dumps(line))
        return 0
    if a.workload == "serving":
        return run_serving(a, spd, synth, line, dev)
    if a.workload == "decimated":
        n_dm, n_samp = 2048, 524288
        sp = synth.ska_like(n_dm, n_samp, n_pulses=200, mean=0.0, sd=1.0, drift_amp=0.0,
                            fwhm_range=(1.0, 400.0), device=dev, seed=1611_6)
        x = sp.data
        n = n_dm * n_samp
        levels = [(0, list(range(1, 33)))] + [(l, list(range(17, 33))) for l in range(1, 5)]
        cap = 1 << 24
        out = torch.empty((cap, 4), dtype=torch.int32, device=dev)
        res = torch.zeros(16, dtype=torch.uint8, device=dev)
        msd = torch.empty(len(levels) * 40, dtype=torch.uint8, device=dev)
        ws = torch.empty(spd.search_decimated_workspace_bytes(x, levels), dtype=torch.uint8,
                         device=dev)
        step = lambda: spd.search_decimated(x, levels, THRESHOLD, cap, out=out, result=res,
                                            msd_out=msd, workspace=ws)
        ms, clocks = timed(step, a.steps, a.warmup, 0)
        cnt = spd.read_result(res)[0]
        plain_w = list(range(1, 513))
        ws2 = torch.empty(spd.search_workspace_bytes(x, plain_w, THRESHOLD), dtype=torch.uint8,
                          device=dev)
        step2 = lambda: spd.search(x, plain_w, THRESHOLD, cap, out=out, result=res,
                                   msd_out=msd[:40], workspace=ws2)
        ms2, _ = timed(step2, max(3, a.steps // 4), 3, 0)
        cnt2 = spd.read_result(res)[0]
        line.update(value=n / (ms / 1e3), ms_per_step=ms, dtype="f32", clocks=clocks,
                    candidates_per_step=cnt, gpu_launches=(5 + 2 * len(levels)) * a.steps,
                    plain_search={"widths": "1..512", "ms_per_step": ms2, "value": n / (ms2 / 1e3),
                                  "candidates": cnt2},
                    roofline=hbm_roofline("decimated step (level planes, per-level MSD, one "
                                          "search launch per level class)",
                                          2 * 4 * n + 16 * cnt, ms,
                                          note="algorithmic bytes of the native plane only"),
                    speedup_vs_plain=ms2 / ms,
                    realtime_factor=n_samp * SAMPLE_TIME_S / (ms / 1e3),
                    config={"workload": f"{n_dm} DM x {n_samp} FP32 N(0,1) + 200 Gaussian pulses "
                                        "(FWHM 1..400); levels 0: widths 1..32, 1-4: 17..32 "
                                        "level samples (native to 512), each level its own "
                                        "MSD; f_T 7",
                            "l2": "inputs larger than L2"})
        print(json.dumps(line))
        return 0
    if a.workload == "plane":
        n_dm, n_samp = a.n_dm, a.n_samp
        x = synth.ska_like(n_dm, n_samp, device=dev, seed=1611_1).data
        n = n_dm * n_samp
        m = spd.msd(x)
        snr = torch.empty((n_dm, n_samp), dtype=torch.float32, device=dev)
        wid = torch.empty((n_dm, n_samp), dtype=torch.int16, device=dev)
        cap = int(n * 0.45) + 1024
        out = torch.empty((cap, 4), dtype=torch.int32, device=dev)
        res = torch.zeros(16, dtype=torch.uint8, device=dev)
        phases = [lambda: spd.boxcar_snr(x, m, WIDTHS, snr_out=snr, width_out=wid),
                  lambda: spd.threshold_candidates(snr, wid, THRESHOLD, cap, out=out, result=res)]
        ms, (box_ms, thr_ms), clocks = timed_split(phases, a.steps, a.warmup, 0)
        cnt = spd.read_result(res)[0]
        n_eval = len(WIDTHS) + (WIDTHS[0] != 1)
        line.update(value=n / (ms / 1e3), ms_per_step=ms, dtype="f32", clocks=clocks,
                    candidates_per_step=cnt, gpu_launches=3 * a.steps,
                    step_breakdown_ms={"boxcar_snr": box_ms, "threshold_candidates": thr_ms},
                    # every width of every sample: add, multiply by 1/sigma_w, max
                    roofline=alu_roofline("boxcar_snr plane kernel (every width, no pruning)",
                                          3.0 * n * n_eval + 5.0 * n, box_ms,
                                          note="3 FP32 operations per (sample, width) + 5 per "
                                               "sample"),
                    hbm_roofline_boxcar=hbm_roofline("boxcar_snr plane kernel", 4 * n + 6 * n,
                                                     box_ms),
                    threshold_roofline=hbm_roofline("threshold_kernel", 6 * n + 16 * cnt, thr_ms),
                    config={"workload": f"unfused calls on the SKA-like chunk {n_dm} x {n_samp} "
                                        "FP32: spd_boxcar_snr (widths 1..16 + 24..256/8) then "
                                        "spd_threshold_candidates (f_T 7)",
                            "l2": "inputs larger than L2"})
        print(json.dumps(line))
        return 0
    if a.workload == "dedisperse":
        n_chan, n_dm = 256, 256
        dms = np.linspace(0.0, 100.0, n_dm)
        delays_np = synth.dispersion_delays(n_chan, dms)
        n_out = 1 << 18
        fb = synth.filterbank(n_chan, n_out + int(delays_np.max()), dms=dms,
                              pulses=((100, 5000, 8, 0.5),), device=dev, seed=1611_8)
        delays = torch.from_numpy(fb.delays).to(dev)
        plane = torch.empty((n_dm, n_out), dtype=torch.float32, device=dev)
        step = lambda: spd.dedisperse(fb.data, delays, n_out, out=plane)
        ms, clocks = timed(step, a.steps, a.warmup, 0)
        fb_bytes = fb.data.numel() * 4
        line.update(value=n_dm * n_out / (ms / 1e3), ms_per_step=ms, dtype="f32", clocks=clocks,
                    gpu_launches=a.steps,
                    roofline=lds_roofline("dedisperse_kernel", float(n_dm) * n_out * n_chan, ms,
                                          note="one FP32 add per (DM trial, channel, sample), "
                                               "its operand read from the channel window "
                                               "staged in shared memory"),
                    hbm_roofline=hbm_roofline("dedisperse_kernel", fb_bytes + n_dm * n_out * 4,
                                              ms, note="the filterbank read once and the plane "
                                                       "written"),
                    adds_per_s=n_dm * n_out * n_chan / (ms / 1e3),
                    config={"workload": f"incoherent de-dispersion, {n_chan} channels "
                                        f"1200-1500 MHz at 64 us, {n_dm} DM trials 0..100, "
                                        f"{n_out} output samples, FP32",
                            "l2": "filterbank %.2f GB" % (fb_bytes / 1e9)})
        print(json.dumps(line))
        return 0
    if a.workload == "cluster":
        n_dm, n_samp = a.n_dm, a.n_samp
        sp = synth.ska_like(n_dm, n_samp, device=dev, seed=1611_1)   # the headline plane
        m = spd.msd(sp.data)
        snr, w = spd.boxcar_snr(sp.data, m, WIDTHS)
        del sp
        torch.cuda.empty_cache()
        cap, gap = 1 << 24, 16
        out = torch.empty((cap, 8), dtype=torch.int32, device=dev)
        res = torch.zeros(16, dtype=torch.uint8, device=dev)
        step = lambda: spd.cluster_rows(snr, w, THRESHOLD, gap, cap, out=out, result=res)
        ms, clocks = timed(step, a.steps, a.warmup, 0)
        cnt, st = spd.read_result(res)
        if st != 0:
            raise RuntimeError(f"cluster status {st}")
        n = n_dm * n_samp
        alg = 6 * n + 32 * min(cnt, cap)   # SNR + width read once, records written
        ach = alg / (ms / 1e3) / 1e9
        line.update(value=n / (ms / 1e3), ms_per_step=ms, dtype="f32", clocks=clocks,
                    clusters_per_step=cnt, gpu_launches=a.steps,
                    roofline={"bound": "hbm", "kernel": "cluster_kernel", "achieved": ach,
                              "peak": hbm, "unit": "GB/s", "frac": ach / hbm, "traffic": None,
                              "peak_source": f"{peak_kind} hbm_gbs",
                              "algorithmic_bytes": alg},
                    config={"workload": f"per-DM clustering (max gap {gap} samples) of the "
                                        f"candidates of the SKA-like {n_dm} x {n_samp} SNR "
                                        "plane (spd_boxcar_snr: widths 1..16 + 24..256/8, "
                                        "f_T 7)",
                            "l2": "inputs larger than L2 (SNR + width planes %.1f GB)"
                                  % (6 * n / 1e9)})
        print(json.dumps(line))
        return 0
    raise SystemExit(f"unknown workload {a.workload}")


def run_serving(a, spd, synth, line, dev):
    """Beams of FP16 chunks served with continuous batching: saturated
    throughput (every chunk queued at the start) and latency under a
    time-compressed real-time arrival schedule."""
    import torch

    from paper_1611_09704_gb300 import serving
    n_dm, widths, thr = 2048, list(range(1, 129)), 7.0
    beams = synth.serving_beams(a.beams, n_dm, a.chunks_per_beam, device=dev, pin_memory=True)
    max_chunk = max(max(b.lengths) for b in beams)
    srv = serving.Server(n_dm, widths, thr, max_chunk, dtype=spd.F16, capacity=1 << 20,
                         host_records=4096, n_slots=a.slots,
                         mem_budget=int(a.mem_budget_gb * 2**30), device=str(dev))

    def schedule(compress, beam_base=0, first_only=False):
        chunks = []
        for b in beams:
            bid = beam_base + b.beam
            srv.add_beam(bid)
            t = 0
            items = list(zip(b.chunks, b.lengths))[: 1 if first_only else None]
            for k, (c, L) in enumerate(items):
                t += L
                chunks.append(serving.Chunk(bid, k, c, L, arrival=t * SAMPLE_TIME_S / compress,
                                            deadline=L * SAMPLE_TIME_S / compress))
            chunks.append(serving.Chunk(bid, len(items), None, 0, arrival=chunks[-1].arrival,
                                        flush=True))
        return chunks

    def drop(chunks):
        for bid in sorted({c.beam for c in chunks}):
            srv.remove_beam(bid)

    for w in range(max(1, min(a.warmup, 3))):           # kernels loaded, pools warm
        ch = schedule(1.0, beam_base=1000 * (w + 1), first_only=True)
        srv.serve(ch, realtime=False)
        drop(ch)
    torch.cuda.synchronize()
    ch = schedule(1.0, beam_base=0)
    clk = Clocks(0)
    sat = serving.summarize(srv.serve(ch, realtime=False), n_dm)
    clocks = clk.stop()
    inflight_sat = srv.scheduler.max_inflight
    drop(ch)
    ch = schedule(a.compress, beam_base=100)
    rt_res = srv.serve(ch, realtime=True)
    rt = serving.summarize(rt_res, n_dm)
    drop(ch)
    n_chunks = sum(len(b.lengths) for b in beams)
    line.update(value=sat["samples_per_s"], ms_per_step=sat["span_s"] * 1e3, dtype="f16",
                clocks=clocks, steps=1, warmup=max(1, min(a.warmup, 3)),
                roofline=hbm_roofline("serving pass (H2D + running MSD + search per chunk)",
                                      2 * 2 * sat["samples"] + 16 * sat["candidates"],
                                      sat["span_s"] * 1e3,
                                      note="host-driven pass timed by wall clock: bounded by "
                                           "the scheduler and host link, not one kernel"),
                candidates_per_step=sat["candidates"],
                # push: MSD, merge, screen, search and the halo out (and in,
                # but for a beam's first); reset and flush: 5
                gpu_launches=n_chunks * 6 + len(beams) * 4,
                saturated=dict(sat, max_inflight=inflight_sat),
                realtime=dict(rt, compress=a.compress, max_inflight=srv.scheduler.max_inflight),
                realtime_factor=sat["samples"] / n_dm * SAMPLE_TIME_S / sat["span_s"],
                config={"workload": f"{a.beams} beams x {a.chunks_per_beam} chunks of {n_dm} DM x "
                                    "U{8192..65536} samples, FP16 N(0,1), Poisson top-hat pulses "
                                    "(0.5/s, SNR U(6,40), width U{1..128}); widths 1..128; f_T 7; "
                                    "running MSD + halo on device; chunks from page-locked host "
                                    "memory (H2D inside every latency)",
                        "slots": a.slots, "mem_budget_gb": a.mem_budget_gb,
                        "samples": sat["samples"], "l2": "inputs larger than L2"})
    print(json.dumps(line))
    return 0


def main():
    a = parse()
    if a.workload != "ska" and a.impl == "spd":
        # single-GPU measurements: under torchrun, rank 0 alone runs them
        if int(os.environ.get("RANK", "0")) != 0:
            return 0
        return run_other(a)
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if a.impl == "reference":
        return run_reference(a, rank, world)
    if world > 1:
        import torch
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    rc = run_spd(a, rank, world, local)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()
    return rc


if __name__ == "__main__":
    sys.exit(main())
