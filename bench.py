"""Throughput benchmark of the GB300 LBM-RANS step.

Workload: NACA 0012 at alpha = 10 deg, Re = 6e6, Ma = 0.15, six 2:1 levels with the
finest spacing c/4096 (coarse h0 = c/128 over an 8c x 4c box, about 1.5M nodes),
FP32 populations and nu_tilde, SA-neg, virtual-node wall function.  One step is one
coarse time step: 2^l sub-steps of every level l, each with its wall function (finest
level), SA-neg update, stream-collide with the cut-link bounce-back and the Rohde
transfers.  The geometry is built once; inputs are synthetic (analytic NACA section).

Metric: MLUPS = sum_l (active nodes of level l) * 2^l per coarse step / time.

Arms:
  default            the CUDA library (one replica per rank under torchrun, no collective)
  --impl reference   the FP64 CPU oracle on the host cores (rank 0 only)

Launch variant: lbm_autotune picks each level's warps per block and PDL on/off from timed
steps before the warm-up (--no-autotune keeps the default variant).

Timing: W untimed warm-up steps, then K steps timed with CUDA events on the solver's
stream; a 512 MB buffer is written between timed steps to flush L2 (the flush is
outside the events).  The dominant kernel's roofline comes from a per-launch event
pass over the same workload right after the timed region.
"""
from __future__ import annotations

import argparse
import json
import platform
import os
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

from paper_2601_18443_gb300 import workloads as W  # noqa: E402

METRIC = "MLUPS"
WORKLOAD = "naca0012_a10_re6e6_ma015_6lvl_c4096"
WORKLOAD_HL = "highlift_3element_a8_re9e6_ma02_8lvl_c8192"
CPU_SAMPLE = "naca0012_a0_re1e6_ma01_6lvl_c256"


def ncu_traffic(key):
    """DRAM bytes of one launch from the committed ncu summary, or None when the kernel
    source changed since the capture."""
    import hashlib
    try:
        vals = {}
        with open(os.path.join(ROOT, "profiles", "dram_traffic.txt")) as f:
            for ln in f:
                if ln.strip() and not ln.startswith("#"):
                    k, v = ln.split()
                    vals[k] = v
        src = os.path.join(ROOT, "paper_2601_18443_gb300", "csrc", "level.cuh")
        with open(src, "rb") as f:
            if hashlib.sha256(f.read()).hexdigest() != vals["level_cuh_sha256"]:
                return None
        return int(vals[key])
    except Exception:
        return None


def method_bytes(store, turbulence):
    """Algorithmic bytes of the method per node update: the stream-collide moves 9 populations
    in and out, reads chi and writes rho and u (88 B in FP32, 52 B with 16-bit storage); SA-neg
    adds chi read and written, u and 1/d^2 read (20 B).  The general form of the
    kernel also reads each cell's flag word, which lbm_get_info counts in its
    bytes_per_node_update; blocks of plain cells read no flag word and, laminar, no chi."""
    pop = 4 if store == 0 else 2
    return 18 * pop + 4 + 12 + (20 if turbulence else 0)


def l2_copy_gbs(dev, mb=24, reps=40, replays=5):
    """Copy bandwidth (read + write) of a working set that stays in L2: two 24 MB buffers
    copied back and forth, reps pairs of copies captured in one CUDA graph (so that launch
    gaps do not count), timed with CUDA events over several replays after a warm-up."""
    import torch
    a = torch.empty(mb << 20, dtype=torch.uint8, device=dev)
    b = torch.empty_like(a)
    side = torch.cuda.Stream(dev)
    side.wait_stream(torch.cuda.current_stream(dev))
    with torch.cuda.stream(side):
        for _ in range(4):
            b.copy_(a); a.copy_(b)
    torch.cuda.current_stream(dev).wait_stream(side)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for _ in range(reps):
            b.copy_(a); a.copy_(b)
    g.replay()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record()
    for _ in range(replays):
        g.replay()
    e1.record()
    torch.cuda.synchronize()
    return replays * reps * 2 * 2 * (mb << 20) / (e0.elapsed_time(e1) * 1e-3) / 1e9


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            p = json.load(f)
        return float(p["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


# --------------------------------------------------------------------------- clocks

class ClockSampler:
    """nvidia-smi samples (every 200 ms) of the SM clock and throttle reasons."""

    FIELDS = ("uuid,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")

    def __init__(self, uuid):
        self.uuid = uuid
        self.proc = None
        self.lines = []
        self.thread = None

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                                          "-lms", "200"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None
            return
        self.thread = threading.Thread(target=self._read, daemon=True)
        self.thread.start()

    def _read(self):
        for ln in self.proc.stdout:
            self.lines.append(ln.strip())

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        if self.thread:
            self.thread.join(timeout=2)
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 8:
                continue
            if self.uuid and parts[0] != self.uuid:
                continue
            try:
                sm.append(float(parts[1]))
                mx.append(float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[4:8]):
                if v.lower() == "active":
                    reasons.add(nm)
        if not sm:
            return None
        return {"sm_mhz": float(np.median(sm)), "sm_max_mhz": float(max(mx)), "reasons": sorted(reasons),
                "samples": len(sm)}


# --------------------------------------------------------------------------- oracle arm

def run_oracle_sample(steps, warmup):
    """Times the FP64 oracle on the host cores; returns (MLUPS, cores, sample text)."""
    import oracle

    cfg, loops = W.naca0012_small()
    s = oracle.Solver(cfg)
    s.set_geometry(loops)
    nu = 0
    for l in range(cfg["levels"]):
        m = s.get_fields(l)["mask"]
        nu += int(((m == 1) | (m == 2)).sum()) << l
    s.step(warmup)
    t0 = time.perf_counter()
    s.step(steps)
    dt = time.perf_counter() - t0
    s.close()
    mlups = nu * steps / dt / 1e6
    sample = (f"{CPU_SAMPLE}: NACA 0012 6 levels to c/256 (coarse 128x64 over 16c x 8c), "
              f"{nu} node updates per coarse step, {steps} coarse steps after {warmup} warm-up, FP64 oracle, "
              f"{dt:.2f} s")
    return mlups, oracle.threads(), sample, dt


def _host_cpu():
    """The host's CPU model as /proc/cpuinfo names it (x86 'model name', else Arm part)."""
    try:
        txt = open("/proc/cpuinfo").read()
        for key in ("model name", "Model", "CPU part"):
            for ln in txt.splitlines():
                if ln.split(":")[0].strip() == key:
                    return f"{key}: {ln.split(':', 1)[1].strip()}"
    except OSError:
        pass
    return platform.processor() or platform.machine()


def oracle_timing(args):
    """The FP64 oracle's node-update rate on this host's cores: config[0] (6 levels to c/256)
    over --oracle-steps0 coarse steps with all threads and with one, and with --oracle-full
    the bench workload (6 levels to c/4096) over --oracle-steps1 coarse steps with all threads
    (its grid build timed apart).  One JSON line; no GPU."""
    import oracle

    oracle.build()
    allt = oracle.threads()
    out = {"metric": "oracle_MLUPS", "unit": "MLUPS", "dtype": "f64", "host": _host_cpu(),
           "machine": platform.machine(), "nproc": os.cpu_count(), "runs": []}

    def run(cfg, loops, name, steps, threads):
        oracle.set_threads(allt)
        t0 = time.perf_counter()
        s = oracle.Solver(cfg)
        s.set_geometry(loops)
        tg = time.perf_counter() - t0
        nu = 0
        for l in range(cfg["levels"]):
            m = s.get_fields(l)["mask"]
            nu += int(((m == 1) | (m == 2)).sum()) << l
        oracle.set_threads(threads)
        s.step(1)
        t0 = time.perf_counter()
        s.step(steps)
        dt = time.perf_counter() - t0
        s.close()
        oracle.set_threads(allt)
        out["runs"].append({"workload": name, "threads": threads, "coarse_steps": steps,
                            "node_updates_per_step": nu, "seconds": round(dt, 2),
                            "mlups": round(nu * steps / dt / 1e6, 3), "geometry_s": round(tg, 1)})
        print(json.dumps(out["runs"][-1]), file=sys.stderr, flush=True)

    cfg0, loops0 = W.naca0012_small()
    run(cfg0, loops0, CPU_SAMPLE, args.oracle_steps0, allt)
    run(cfg0, loops0, CPU_SAMPLE, args.oracle_steps0, 1)
    if args.oracle_full:
        cfg1, loops1 = W.naca0012_large()
        run(cfg1, loops1, WORKLOAD, args.oracle_steps1, allt)
    print(json.dumps(out), flush=True)
    return 0


def reference_arm(args, rank, world):
    if rank != 0:
        return 0
    steps = max(1, args.steps)
    mlups, cores, sample, dt = run_oracle_sample(steps, max(0, min(args.warmup, 3)))
    line = {
        "impl": "reference", "metric": METRIC, "value": round(mlups, 4), "unit": "MLUPS", "n_gpus": 0,
        "steps": steps, "warmup": args.warmup, "ms_per_step": round(1e3 * dt / steps, 3),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": WORKLOAD, "arm": "FP64 CPU oracle on host cores (bounded sample)",
                   "sample": f"each step is one coarse step of {CPU_SAMPLE} (the same multilevel method at "
                             f"c/256, 207k node updates): the oracle's node-update rate stands for the workload's, "
                             f"whose 21.4M node updates per coarse step would take seconds each"},
        "cpu_baseline": {"value": round(mlups, 4), "unit": "MLUPS", "cores": cores, "kind": "oracle",
                         "sample": sample},
        "e2e": {"value": round(mlups, 4), "unit": "MLUPS", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


# --------------------------------------------------------------------------- replicas

def replica_totals(ms, units, dist, device):
    """Whole-job timing of independent replicas: the slowest rank's time and the sum of
    the node updates of all ranks (no collective touches the solver's data)."""
    if dist is None:
        return ms, units
    import torch
    t = torch.tensor([ms], dtype=torch.float64, device=device)
    u = torch.tensor([float(units)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    dist.all_reduce(u, op=dist.ReduceOp.SUM)
    return float(t.item()), float(u.item())


# --------------------------------------------------------------------------- GPU arm

def gpu_arm(args, rank, world, dist):
    import torch

    import paper_2601_18443_gb300 as pkg

    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    pkg.library()
    # a dedicated stream (the legacy default stream has handle 0, which the library
    # would replace by a stream of its own): events and steps share this stream
    stream = torch.cuda.Stream(dev)
    torch.cuda.set_stream(stream)
    hl = args.workload == "highlift"
    tune_steps = 10
    if hl:
        # three-element high-lift case, 8 levels to c/8192 (555M node updates per coarse
        # step, 22 ms each): a few timed steps; the extra measurements are skipped.  Started
        # impulsively it diverges after about 35 coarse steps, so the autotuner times one
        # coarse step per candidate on a checkpoint of the initial state, the solve is
        # rewound to it, and 10 steps are timed after 3 warm-up steps.
        cfg, loops = W.highlift_3element()
        args.steps, args.warmup, tune_steps = min(args.steps, 10), 3, 1
        args.no_cpu_baseline = args.no_hbm_grid = args.no_precision_forms = True
    else:
        cfg, loops = W.naca0012_large()
    K = args.steps
    s = pkg.Solver(cfg, stream=stream)
    s.set_geometry(loops)
    # launch autotuner (warps per block of each level, PDL on/off);
    # its steps are untimed
    if args.no_autotune:
        tune = None
    elif hl:
        blob = s.get_state()
        tune = s.autotune(tune_steps)
        s.set_state(blob)        # the tuned launch form stays; the steps start again from 0
    else:
        tune = s.autotune(tune_steps)
    info = s.info()
    nu_step = info["node_updates_per_step"]
    flush = torch.empty(512 << 20, dtype=torch.uint8, device=dev)

    s.step(args.warmup)
    torch.cuda.synchronize()
    K = args.steps
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(K)]
    uuid = None
    try:
        uuid = "GPU-" + str(torch.cuda.get_device_properties(dev).uuid)
    except Exception:
        pass
    clocks = ClockSampler(uuid)
    clocks.start()
    time.sleep(0.5)
    if dist is not None:
        dist.barrier()
    torch.cuda.synchronize()
    for k in range(K):
        flush.fill_(k & 0xFF)
        ev[k][0].record(stream)
        s.step_async(1)
        ev[k][1].record(stream)
    torch.cuda.synchronize()
    if dist is not None:
        dist.barrier()
    clk = clocks.stop()
    s.synchronize()          # status word: non-finite fields raise here
    ms = sum(a.elapsed_time(b) for a, b in ev)
    ms, units = replica_totals(ms, nu_step * K, dist, dev)
    value = units / (ms * 1e-3) / 1e6

    # dominant kernel: per-launch CUDA events on the solver stream over the same workload
    kt = s.time_kernels(max(2, min(10, K)))
    fin = kt["level_step_finest"]
    avg_ms = fin["ms"] / max(fin["launches"], 1)
    act_fin = info["cells_active"][-1]
    bpn_kernel = info["bytes_per_node_update"]
    bpn = method_bytes(cfg.get("store", 0), cfg.get("turbulence", 0))
    achieved = act_fin * bpn / (avg_ms * 1e-3) / 1e9
    peak, peak_kind = peaks()
    l2_peak = l2_copy_gbs(dev) if rank == 0 else None
    total_kt = sum(v["ms"] for v in kt.values())
    # the same launches inside the step graphs (per-block global-timer records, after the
    # timed region): first block past its wait to last block done, per launch
    s.set_timeline(True)
    s.step(4)
    tl = s.timeline()
    s.set_timeline(False)
    L_ = info["levels"]
    fin_tl = [e["t_end_us"] - e["t_wait_us"] for e in tl if e["level"] == L_ - 1 and e["kind"] in (0, 1)]
    in_graph_us = float(np.mean(fin_tl)) if fin_tl else None
    breakdown = {}
    for g in (0, 1):
        evg = [e for e in tl if e["graph"] == g]
        if not evg:
            continue
        span = max(e["t_end_us"] for e in evg)
        cls = {"finest": 0.0, "coarser": 0.0, "prolong": 0.0}
        for e in evg:
            key = "prolong" if e["kind"] == 2 else ("finest" if e["level"] == L_ - 1 else "coarser")
            cls[key] += e["t_end_us"] - e["t_wait_us"]
        cls["between_launches"] = span - sum(cls.values())
        cls["graph_span"] = span
        for key, v in cls.items():
            breakdown[key] = breakdown.get(key, 0.0) + v / 2
    loads = s.get_loads()

    # end to end through the public API: host polyline -> grid build + upload -> K steps -> loads to host
    e2e = None
    if rank == 0 or world > 1:
        xy_bytes = sum(np.asarray(p).nbytes for p in loops) + 4 * (len(loops) + 1)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        s2 = pkg.Solver(cfg, stream=stream)
        ta = time.perf_counter()
        s2.set_geometry(loops)
        tb = time.perf_counter()
        s2.step(K)
        tc = time.perf_counter()
        l2 = s2.get_loads()
        t1 = time.perf_counter()
        dev_b = s2.info()["device_bytes"]
        s2.close()
        n_seg = len(l2["cp"])
        e2e = {"value": round(nu_step * K / (t1 - t0) / 1e6, 2), "unit": "MLUPS",
               "h2d_bytes_per_step": int((xy_bytes + dev_b) / K),
               "d2h_bytes_per_step": int((56 + 16 * n_seg) / K),
               "what": f"lbm_create + lbm_set_geometry (host grid build, table upload) + lbm_step({K}) + "
                       f"lbm_get_loads, wall clock; h2d counts the polyline plus the uploaded tables "
                       f"(upper bound: device bytes held) spread over the K steps",
               "phases_s": {"create": round(ta - t0, 4), "set_geometry": round(tb - ta, 4),
                            "steps": round(tc - tb, 4), "loads": round(t1 - tc, 4)}}
        # the host-only part of set_geometry (grid build and table fill), timed apart
        tp = time.perf_counter()
        pkg.plan(cfg, loops)
        e2e["host_grid_build_s"] = round(time.perf_counter() - tp, 4)

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        mlups_c, cores, sample, _ = run_oracle_sample(args.cpu_steps, 2)
        cpu = {"value": round(mlups_c, 4), "unit": "MLUPS", "cores": cores, "kind": "oracle", "sample": sample}

    hbm = hbm_sc = None
    if rank == 0 and not args.no_hbm_grid:
        hbm = hbm_grid_roofline(pkg, stream, peak, peak_kind, tune=not args.no_autotune)
        hbm_sc = hbm_grid_roofline(pkg, stream, peak, peak_kind, turbulence=0, tune=not args.no_autotune)

    # precision forms: the same workload with populations stored in FP16 / BF16
    forms = None
    if rank == 0 and not args.no_precision_forms:
        forms = {}
        for name, store in (("fp16", 1), ("bf16", 2)):
            c2 = dict(cfg)
            c2["store"] = store
            s3 = pkg.Solver(c2, stream=stream)
            s3.set_geometry(loops)
            s3.step(args.warmup)
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            kk = max(10, K // 2)
            msum = 0.0
            for _ in range(kk):
                flush.fill_(1)
                e0.record(stream)
                s3.step_async(1)
                e1.record(stream)
                torch.cuda.synchronize()
                msum += e0.elapsed_time(e1)
            s3.synchronize()
            kt3 = s3.time_kernels(3)
            f3 = kt3["level_step_finest"]
            avg3 = f3["ms"] / max(f3["launches"], 1)
            bpn3 = method_bytes(store, 1)
            forms[name] = {"value": round(nu_step * kk / (msum * 1e-3) / 1e6, 2), "unit": "MLUPS",
                           "ms_per_step": round(msum / kk, 4), "bytes_per_node_update": bpn3,
                           "finest_kernel_gbs": round(act_fin * bpn3 / (avg3 * 1e-3) / 1e9, 1)}
            s3.close()
            # the same storage on the HBM-bound 4096^2 level (SA on), against FP32 there
            g16 = hbm_grid_roofline(pkg, stream, peak, peak_kind, tune=not args.no_autotune, store=store)
            forms[name]["hbm_grid_mlups"] = g16["mlups"]
            forms[name]["hbm_grid_frac"] = g16["frac"]
            sc16 = hbm_grid_roofline(pkg, stream, peak, peak_kind, turbulence=0, tune=not args.no_autotune, store=store)
            forms[name]["stream_collide_mlups"] = sc16["mlups"]
            forms[name]["stream_collide_frac"] = sc16["frac"]

    if rank == 0:
        line = {
            "metric": METRIC, "value": round(value, 2), "unit": "MLUPS", "n_gpus": world, "steps": K,
            "warmup": args.warmup, "ms_per_step": round(ms / K, 4), "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": WORKLOAD_HL if hl else WORKLOAD, "nodes": int(sum(info["cells_active"])),
                       "node_updates_per_step": int(nu_step), "levels": info["levels"],
                       "cells_active_per_level": [int(x) for x in info["cells_active"]],
                       "l2": "512 MB buffer written between timed steps (outside the events)",
                       "replicas": world, "parallelism": f"replicas{world}"},
            "gbs_full_step_algorithmic": round(value * 1e6 * bpn / 1e9, 1),
            "bytes_per_node_update": {"method": bpn, "kernel": bpn_kernel},
            "roofline": {"bound": "hbm", "achieved": round(achieved, 1), "peak": peak, "unit": "GB/s",
                         "frac": round(achieved / peak, 4), "traffic": None if hl else ncu_traffic("workload_finest_launch"),
                         "kernel": "k_level (finest level: wall function + SA-neg + stream-collide)", "peak_kind": peak_kind,
                         "bytes_per_node_update": bpn, "bytes_per_launch": int(act_fin * bpn),
                         "avg_launch_ms": round(avg_ms, 5),
                         "share_of_step": round(fin["ms"] / total_kt, 3) if total_kt > 0 else None,
                         "kernel_bytes_per_node_update": bpn_kernel,
                         "frac_kernel_bytes": round(act_fin * bpn_kernel / (avg_ms * 1e-3) / 1e9 / peak, 4),
                         "in_graph": None if in_graph_us is None else {
                             "avg_launch_us": round(in_graph_us, 2),
                             "achieved": round(act_fin * bpn / (in_graph_us * 1e-6) / 1e9, 1),
                             "frac": round(act_fin * bpn / (in_graph_us * 1e-6) / 1e9 / peak, 4),
                             "how": "the same launches inside the step graphs: first block past its wait for the "
                                    "preceding kernel to last block done (lbm_get_timeline, global timer); "
                                    "avg_launch_ms above brackets each launch with CUDA events outside the graphs"}},
            "step_breakdown_us": {k: round(v, 1) for k, v in breakdown.items()} or None,
            "roofline_l2": None if l2_peak is None else {
                "bound": "l2", "achieved": round(achieved, 1), "peak": round(l2_peak, 1), "unit": "GB/s",
                "frac": round(achieved / l2_peak, 4),
                "l2_bytes": None if hl else ncu_traffic("workload_finest_launch_lts"),
                "kernel": "k_level (finest level)",
                "peak_kind": "measured in this run: copies of a 48 MB working set that stays in L2 (graph-replayed)",
                "why": "the finest level's state (tens of MB) is largely served by L2 between its sub-steps"},
            "kernel_times": {k: {"ms_per_step": round(v["ms"] / max(2, min(10, K)), 4), "launches": v["launches"]}
                             for k, v in kt.items()},
            "gpu_launches": int(info["kernels_per_step"] * K),
            "clocks": clk,
            "loads": {"CL": loads["CL"], "CD": loads["CD"], "step": loads["step"]},
            "e2e": e2e,
            "autotune": None if tune is None else {
                "min_blocks_per_level": tune["min_blocks"], "sched_per_level": tune["sched"],
                "shape_per_level": tune["shape"],
                "pdl": tune["pdl"],
                "step_us_default": round(tune["default_step_us"], 2),
                "step_us_tuned": round(min(tune["step_us"].values()), 2)},
        }
        if cpu is not None:
            line["cpu_baseline"] = cpu
        if hbm is not None:
            line["roofline_hbm_grid"] = hbm
            line["roofline_stream_collide"] = hbm_sc
        if forms is not None:
            line["precision_forms"] = forms
        print(json.dumps(line), flush=True)
    s.close()
    return 0


def hbm_grid_roofline(pkg, stream, peak, peak_kind, n=4096, turbulence=1, tune=True, store=0):
    """The level kernel on one periodic 4096 x 4096 level (1.4-1.7 GB of traffic per
    launch, far beyond L2): its HBM roofline without multilevel effects; turbulence=0
    leaves the stream-collide alone (88 B per node update in FP32)."""
    cfg = W.base_config(levels=1, nx0=n, ny0=n, h0=1.0, Re=1000.0, Ma=0.1, periodic=1, solid_walls=0,
                        turbulence=turbulence, wall_model=3, store=store)
    s = pkg.Solver(cfg, stream=stream)
    s.set_geometry([])
    if tune:
        s.autotune(3)
    s.step(3)
    kt = s.time_kernels(5)
    info = s.info()
    sc = kt["level_step_finest"]
    avg = sc["ms"] / sc["launches"]
    cells = info["cells_active"][0]
    bpn = method_bytes(store, turbulence)
    bpl = cells * bpn
    # every block of the periodic level is plain: no flag word, and chi only with SA-neg
    bpk = info["bytes_per_node_update"] - (4 if turbulence else 8)
    s.close()
    ach = bpl / (avg * 1e-3) / 1e9
    return {"bound": "hbm", "achieved": round(ach, 1), "peak": peak, "unit": "GB/s", "frac": round(ach / peak, 4),
            "traffic": (ncu_traffic("hbm_grid_launch" if turbulence else "stream_collide_launch") if not store else None),
            "kernel": "k_level", "grid": f"{n}x{n} periodic, 1 level, SA {'on' if turbulence else 'off'}",
            "bytes_per_node_update": bpn, "bytes_per_launch": int(bpl),
            "kernel_bytes_per_node_update": bpk,
            "frac_kernel_bytes": round(cells * bpk / (avg * 1e-3) / 1e9 / peak, 4),
            "avg_launch_ms": round(avg, 4), "mlups": round(cells / avg / 1e3, 1),
            "peak_kind": peak_kind}


def profile_case(args):
    """Small cases for ncu captures: 'hbm_grid' (one periodic 4096 x 4096 level) or
    'workload' (the benchmark workload); a few steps each, no timing."""
    import torch

    import paper_2601_18443_gb300 as pkg

    torch.cuda.set_device(0)
    if args.profile_case in ("hbm_grid", "hbm_grid_laminar"):
        cfg = W.base_config(levels=1, nx0=4096, ny0=4096, h0=1.0, Re=1000.0, Ma=0.1, periodic=1, solid_walls=0,
                            turbulence=int(args.profile_case == "hbm_grid"), wall_model=3)
        loops = []
    else:
        cfg, loops = W.naca0012_large()
    s = pkg.Solver(cfg)
    s.set_geometry(loops)
    if args.profile_variant:
        mb, sc, sh = (int(v) for v in args.profile_variant.split(","))
        L = cfg["levels"]
        s.set_launch_variant([mb] * L, 1, [sc] * L, [sh] * L)
    elif not args.no_autotune:
        s.autotune(2)
    # the steps to profile sit in an NVTX range ("steps"): ncu --nvtx --nvtx-include steps/
    torch.cuda.nvtx.range_push("steps")
    s.step(args.steps)
    torch.cuda.nvtx.range_pop()
    if args.timeline:
        # in-graph launch times of the last run of each step graph (lbm_get_timeline)
        s.set_timeline(True)
        s.step(max(args.steps, 2))
        tl = s.timeline()
        L = cfg["levels"]
        for g in (0, 1):
            ev = [e for e in tl if e["graph"] == g]
            if not ev:
                continue
            span = max(e["t_end_us"] for e in ev)
            rows = {}
            for e in ev:
                key = f"prolong from level {e['level']}" if e["kind"] == 2 else f"level {e['level']} {'odd' if e['kind'] else 'even'}"
                r = rows.setdefault(key, [0, 0.0])
                r[0] += 1
                r[1] += e["t_end_us"] - e["t_wait_us"]
            busy = sum(r[1] for r in rows.values())
            print(f"timeline graph {g}: span {span:.1f} us, launches {len(ev)}, between launches {span - busy:.1f} us")
            for key in sorted(rows):
                n, t = rows[key]
                print(f"  {key:26s} launches {n:3d}  total {t:8.1f} us  mean {t / n:6.2f} us")
    print("profile case", args.profile_case, "ok", flush=True)
    s.close()
    return 0


def serving_arm(args):
    """Continuous batching of the seeded polar-request stream (NACA 4-digit sections,
    4..7 levels, Poisson arrivals) against the same stream served one solve at a time."""
    import torch

    import paper_2601_18443_gb300 as pkg
    from paper_2601_18443_gb300.serve import GpuBackend, Service, SolveRequest, summarize

    pkg.library()
    torch.cuda.set_device(0)
    rate = args.serving_rate
    reqs = []
    for q in W.polar_requests(args.serving, rate_per_s=rate if rate > 0 else 2.0):
        cfg, loops = W.polar_case(q)
        reqs.append(SolveRequest(rid=q["rid"], arrival=q["arrival"] if rate > 0 else 0.0, cfg=cfg, loops=loops,
                                 max_steps=args.serving_max_steps, min_steps=args.serving_min_steps,
                                 check_every=100, window=args.serving_window, tol=args.serving_tol, patience=2))
    uuid = None
    try:
        uuid = "GPU-" + str(torch.cuda.get_device_properties(0).uuid)
    except Exception:
        pass
    out = {}
    # batched: resident solves stepped together, one launch per level-schedule node for all of
    # them (lbm_batch); streams: the same slots, each solve on its own stream with its own
    # launches; one_at_a_time: one slot
    arms = [("batched", args.serving_slots, True)]
    if not args.serving_no_baseline:
        arms += [("streams", args.serving_slots, False), ("one_at_a_time", 1, False)]
    if args.serving_arms:
        arms = [a for a in arms if a[0] in args.serving_arms.split(",")]
    clk = None
    for name, slots, batched in arms:
        clocks = ClockSampler(uuid)
        clocks.start()
        svc = Service(max_slots=slots, backend=GpuBackend(), batched=batched)
        res = svc.run(reqs)
        c = clocks.stop()
        if name == "batched":
            clk = c
        sm = summarize(res)
        if args.serving_dump:
            with open(f"{args.serving_dump}.{name}.json", "w") as fh:
                json.dump([dict(rid=r.rid, status=r.status, levels=q.cfg["levels"], arrival=r.arrival,
                                admitted=r.admitted, started=r.started, finished=r.finished, steps=r.steps,
                                history=r.history, message=r.message) for r, q in zip(res, reqs)], fh)
        sm["max_resident"] = max((n for *_, n in svc.trace), default=0)
        sm["clocks"] = c
        out[name] = sm
        by_levels = {}
        for r, q in zip(res, reqs):
            by_levels.setdefault(q.cfg["levels"], []).append(r)
        sm["by_levels"] = {L: dict(n=len(v), steps_mean=float(np.mean([r.steps for r in v])),
                                   latency_p50_s=float(np.median([r.latency for r in v])))
                           for L, v in sorted(by_levels.items())}
    b = out[arms[0][0]]
    line = {"metric": "solves_per_hour", "value": b.get("solves_per_hour"), "unit": "solves/h", "n_gpus": 1,
            "higher_is_better": True, "impl": "ours", "dtype": "f16-store/f32",
            "data": "synthetic", "config": {"workload": f"polar_stream_{args.serving}req_seed2026",
                                           "rate_per_s": rate, "slots": args.serving_slots,
                                           "max_steps": args.serving_max_steps, "min_steps": args.serving_min_steps,
                                           "window_steps": 100 * args.serving_window, "tol_window_mean_CL": args.serving_tol},
            "serving": out, "clocks": clk}
    print(json.dumps(line), flush=True)
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--cpu-steps", type=int, default=300)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-hbm-grid", action="store_true")
    ap.add_argument("--no-precision-forms", action="store_true")
    ap.add_argument("--profile-case", choices=["hbm_grid", "hbm_grid_laminar", "workload"], default=None)
    ap.add_argument("--no-autotune", action="store_true", help="keep the default launch variant")
    ap.add_argument("--oracle-timing", action="store_true",
                    help="time the FP64 oracle on this host's cores (config[0] all threads and one thread; "
                         "with --oracle-full also the bench workload); no GPU")
    ap.add_argument("--oracle-steps0", type=int, default=1000)
    ap.add_argument("--oracle-full", action="store_true")
    ap.add_argument("--oracle-steps1", type=int, default=50)
    ap.add_argument("--timeline", action="store_true",
                    help="profile case: also print the in-graph launch times (lbm_get_timeline) per level")
    ap.add_argument("--profile-variant", default="",
                    help="profile case: launch variant 'min_blocks,sched,shape' on every level (sched 2 two-warp "
                         "blocks, otherwise four-warp blocks) instead of autotuning")
    ap.add_argument("--workload", choices=["naca0012", "highlift"], default="naca0012",
                    help="highlift: the three-element 8-level case (10 timed steps, no extra measurements)")
    ap.add_argument("--serving", type=int, default=0, help="serve this many requests of the polar stream")
    ap.add_argument("--serving-slots", type=int, default=16)
    ap.add_argument("--serving-rate", type=float, default=2.0, help="mean arrivals per second (0: all at once)")
    ap.add_argument("--serving-max-steps", type=int, default=8000)
    ap.add_argument("--serving-min-steps", type=int, default=1600)
    ap.add_argument("--serving-window", type=int, default=8, help="chunks of 100 level-0 steps per CL window")
    ap.add_argument("--serving-tol", type=float, default=5e-3, help="|change of the window-mean CL|")
    ap.add_argument("--serving-no-baseline", action="store_true")
    ap.add_argument("--serving-arms", default="", help="comma list of arms to run: batched,streams,one_at_a_time")
    ap.add_argument("--serving-dump", default=None, help="write per-request results to <path>.<arm>.json")
    args = ap.parse_args()
    if args.oracle_timing:
        return oracle_timing(args)
    if args.profile_case:
        return profile_case(args)
    if args.serving:
        return serving_arm(args)
    if args.warmup < 3 and args.impl == "ours":
        args.warmup = 3
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    if args.impl == "reference":
        return reference_arm(args, rank, world)
    dist = None
    if world > 1:
        import torch
        import torch.distributed as td
        torch.cuda.set_device(int(os.environ.get("LOCAL_RANK", "0")))
        td.init_process_group("nccl")
        dist = td
    rc = gpu_arm(args, rank, world, dist)
    if dist is not None:
        dist.destroy_process_group()
    return rc


if __name__ == "__main__":
    sys.exit(main())
