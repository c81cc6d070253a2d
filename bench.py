#!/usr/bin/env python
"""Benchmark of the GB300 superlattice BTE solver.

One benchmark step is one complete solve of the configured workload through
the C ABI: return to the equilibrium start with the start-up half step
(bte_reset), every leap-frog step of the run (bte_run: one fused kernel per
step, replayed from CUDA graphs), and the window reductions
(bte_observables).  Default workload: the low-temperature single instance
with harmonics n = 0..2048 and 8193 phi_y points on [-80, 80], dt = 2.5e-4,
mu = 20, 30 drive periods (251,340 steps), FP32 state with FP64 reductions:
the largest configuration, whose 537 MB of state streams from HBM every
step.

The metric is cell-updates per second: one cell (n, m) advanced by one full
dt on both the whole and the fractional grid counts once (the paper's MLUPS
convention, Sec. 7).

Multi-GPU (torchrun): every rank solves its own replica; value = all ranks'
cell-updates / the slowest rank's time ("scaling": "weak").  There is no
data-path collective.

``--impl reference`` times the FP64 CPU oracle instead (a bounded sample of
the same workload on the host cores).
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
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "cell-updates/s & sweep points/s at ≤1e-5 abs absorption error; % mem roofline"
UNIT = "cell-updates/s"
PROFILE_FILE = os.path.join(ROOT, "profiles", "pair_step_c3_fp32.md")


def workload(name: str, precision: str):
    from paper_1401_6047_gb300 import workloads as W
    prec = W.FP64 if precision == "fp64" else W.FP32_MIXED
    table = {
        "c1": (W.c1_fp64().replace(precision=prec),
               "single instance: n=0..30, 201 phi_y points on [-10,10], dt=1e-3, mu=1, E_dc=1, "
               "E_omega=0.1, omega=1, B=0, 20 periods"),
        "c2": (W.c2(prec),
               "single instance: n=0..400, 4001 phi_y points on [-40,40], dt=5e-4, mu=2, E_dc=2, "
               "E_omega=0.5, omega=2, B=4, 50 periods, last 10 averaged"),
        "c3": (W.c3(prec),
               "low-temperature single instance: n=0..2048, 8193 phi_y points on [-80,80], "
               "dt=2.5e-4, mu=20, E_dc=4, E_omega=1, omega=3, B=8, 30 periods"),
        "table1": (W.paper_table1(prec),
                   "the paper's Table 1 run: 120 harmonics, 4000 phi_y points on [-6,6], "
                   "dt=1e-4, mu=116, E_dc=7, E_omega=0.1, omega=10, B=4, t=10"),
    }
    return table[name]


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


L2_BYTES = 129 * 1024 * 1024  # GB300 L2

# Observables of full FP64 runs on the GPU (the FP64 path matches the FP64
# oracle to 1e-10 relative wherever the tests can run the oracle); an FP32
# line of the same full run reports its error against them.
FP64_FULL_RUN = {
    "c3": {"absorption": 0.025010811021768893, "v_dc": 0.0614839874218562, "steps": 251340,
           "how": "python -m paper_1401_6047_gb300.precision_study c3 on one GB300 "
                  "(FP64 run: 561 s)"},
}


def measure_l2_gbs(dev, mb: int = 24, reps: int = 50) -> float:
    """Copy bandwidth (read + write bytes) of a buffer pair that fits L2:
    b.copy_(a) over mb MB, repeated back to back after a warm-up, timed with
    CUDA events; the best of 5 rounds.  The roof of a kernel whose state
    stays in L2 between steps."""
    import torch
    n = mb * 1024 * 1024 // 4
    a = torch.ones(n, dtype=torch.float32, device=dev)
    b = torch.empty_like(a)
    for _ in range(10):
        b.copy_(a)
    best = 0.0
    for _ in range(5):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(reps):
            b.copy_(a)
        e1.record()
        torch.cuda.synchronize()
        best = max(best, 2 * 4 * n * reps / (e0.elapsed_time(e1) * 1e-3) / 1e9)
    return best


def kernel_sha() -> str:
    """Hash of the two-step kernel's sources (the kernel file and the device
    helpers and shared declarations it includes)."""
    h = hashlib.sha256()
    for name in ("bte_pair.cu", "bte_device.cuh", "bte_internal.h"):
        with open(os.path.join(ROOT, "paper_1401_6047_gb300", "csrc", name), "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:16]


def single_route(p, elem: int):
    """(kernel, steps per batch of kept rows) that the library chooses for a
    single instance whose launch shape is left to it: "grid_kernel" (on chip,
    one block per SM), "pair_kernel" (two steps per launch) or
    "fused_step_kernel" (one)."""
    from paper_1401_6047_gb300 import bte
    N1, M1 = p.n_max + 1, p.m_points
    row_bytes = 2 * -(-M1 // 32) * 32 * elem
    _, _, K, _ = bte.time_grid(p)
    fits = False
    for V in ((1,) if elem == 8 else (2, 4)):
        for gr in range(1, min(N1, 152) + 1):
            R = -(-N1 // gr)
            W = -(-(-(-M1 // (152 // gr))) // V) * V
            b = ((4 * (R + 2) + 6) * (W + 2 * V) + 2 * (R + 2)) * elem
            fits |= -(-b // 16) * 16 + 16 * (W + 2 + R) + 8 * (-(-W // V) + R) <= 232448
    if fits:
        arr = -(-N1 * bte.launch_shape(p)["pitch"] * elem // 256) * 256
        return "grid_kernel", max(min(min(max(4 * arr, 2 << 20), 16 << 20) // row_bytes, 4096, K), 1)
    if elem == 4:
        return "pair_kernel", max(min((16 << 20) // row_bytes, 4096, K + 3) // 4 * 4, 4)
    return "fused_step_kernel", 0


def ncu_traffic(config_key: str):
    """DRAM bytes per launch of the two-step kernel from the committed ncu
    summary, or None when the summary is missing or the kernel source changed
    since it was taken."""
    try:
        with open(PROFILE_FILE) as f:
            txt = f.read()
    except OSError:
        return None
    sha = None
    val = None
    for line in txt.splitlines():
        line = line.strip().strip("-* ")
        if line.startswith("kernel_sha:"):
            sha = line.split(":", 1)[1].strip()
        if line.startswith(f"traffic_bytes_per_launch[{config_key}]:"):
            try:
                val = float(line.split(":", 1)[1].strip())
            except ValueError:
                val = None
    if sha != kernel_sha():
        return None
    return val


class ClockSampler:
    """nvidia-smi samples of SM clock and throttle reasons during the timed region."""

    FIELDS = ("index,uuid,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, uuid: str | None):
        self.uuid = uuid
        self.proc = None
        self.lines: list[str] = []
        self.thread = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "200"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None
            return
        self.thread = threading.Thread(target=self._read, daemon=True)
        self.thread.start()

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

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
        for line in self.lines:
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 10:
                continue
            if self.uuid and self.uuid not in parts[1]:
                continue
            try:
                sm.append(float(parts[2]))
                mx.append(float(parts[3]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[6:10]):
                if v.lower() == "active":
                    reasons.add(nm)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx),
                "reasons": sorted(reasons), "samples": len(sm)}


def dist_setup():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def oracle_sample(p, target_s: float):
    """Times the oracle as it stands on a bounded number of steps of workload p;
    returns (cell-updates/s, threads, steps, seconds)."""
    import oracle
    st = oracle.init(p)
    t0 = time.perf_counter()
    oracle.advance(p, st, 0, 2)
    dt2 = time.perf_counter() - t0
    n = max(2, min(2000, int(target_s / max(dt2 / 2, 1e-6))))
    t0 = time.perf_counter()
    oracle.advance(p, st, 2, n)
    el = time.perf_counter() - t0
    return p.cells * n / el, oracle.threads(), n, el


def run_reference(args):
    world, rank, _ = dist_setup()
    p, desc = workload(args.config, args.precision)
    if args.periods:
        p = p.replace(periods=args.periods, avg_window=min(p.avg_window, args.periods))
        desc += f" (run shortened to {args.periods:g} periods)"
    if rank != 0:
        return 0
    import oracle
    oracle.build()
    per_step = max(1.0, 60.0 / max(1, args.steps + args.warmup))
    for _ in range(args.warmup):
        oracle_sample(p, min(per_step, 5.0))
    vals, cores, nsteps, secs = [], 0, 0, 0.0
    for _ in range(args.steps):
        v, cores, n, el = oracle_sample(p, per_step)
        vals.append(v)
        nsteps += n
        secs += el
    value = p.cells * nsteps / secs
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * secs / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic",
        "config": {"workload": args.config + ": " + desc, "n_max": p.n_max,
                   "m_points": p.m_points, "precision": "fp64 (oracle)"},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle",
                         "sample": f"{nsteps} leap-frog steps of the {p.n_max + 1}x{p.m_points} "
                                   f"grid from the equilibrium start, in {args.steps} samples"},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


def run_ours(args):
    import torch

    world, rank, local = dist_setup()
    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    dev = torch.device("cuda", torch.cuda.current_device())
    from paper_1401_6047_gb300 import bte

    p, desc = workload(args.config, args.precision)
    if args.periods:
        p = p.replace(periods=args.periods, avg_window=min(p.avg_window, args.periods))
        desc += f" (run shortened to {args.periods:g} periods)"
    dt_eff, P, K, Kw = bte.time_grid(p)
    cells = p.cells
    elem = 8 if args.precision == "fp64" else 4
    stream = torch.cuda.Stream(device=dev)
    state_bytes = 8 * elem * cells  # ping-pong sets of a, b on both grids
    mode = args.mode
    if args.on_chip:
        mode = "on-chip"
    if mode == "auto":
        # the form the library chooses (faster than the persistent mode also
        # where L2 holds the state)
        mode = "streamed"
    resident = {"streamed": 0, "on-chip": 1, "persistent": 2, "on-chip-clusters": 3}[mode]
    on_chip = resident in (1, 3)
    solver = bte.Solver(p, stream=stream.cuda_stream, tile_m=args.tile_m, chunk_n=args.chunk_n,
                        graph_steps=args.graph_steps, vec=args.vec, resident=resident)
    graph_len = min(args.graph_steps or 1024, K)
    if resident == 1:
        # init, start-up half step, step-0 observables; one on-chip launch and
        # the step-counter update; finalize
        launches_per_solve = 3 + 2 + 1
    elif resident == 3:
        # set-up as above; per 8192 steps the on-chip launch over clusters,
        # the fold of its per-cluster sums and a counter update; finalize
        launches_per_solve = 3 + 3 * (-(-K // 8192)) + 1
    elif mode == "persistent":
        # set-up as above; per 8192 steps one persistent launch and a counter
        # update; finalize
        launches_per_solve = 3 + 2 * (-(-K // 8192)) + 1
    else:
        launches_per_solve = 3 + K + (K // graph_len) + (1 if K % graph_len else 0) + 1
    kernel = {"on-chip": "resident_kernel", "persistent": "fused_step_kernel, persistent",
              "on-chip-clusters": "wide_kernel", "streamed": "fused_step_kernel"}[mode]
    if not (args.tile_m or args.chunk_n or args.graph_steps or args.vec) and resident in (0, 3):
        route, batch = single_route(p, elem)
        if route == "grid_kernel":
            # set-up as above; per batch the on-chip launch, the sums of its
            # rows and a counter update; finalize
            kernel, on_chip = route, True
            launches_per_solve = 3 + 3 * (-(-K // batch)) + 1
        elif route == "pair_kernel" and resident == 0:
            # one launch per two steps, per batch the sums and a counter
            # update; an odd last step is one launch and a counter update
            kernel = route
            launches_per_solve = 3 + K // 2 + 2 * (-(-(K // 2 * 2) // batch)) + 2 * (K % 2) + 1

    # L2 flush buffer (larger than the 129 MB L2), written between timed steps
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)

    def one_solve(ev=None):
        if ev:
            ev[0].record(stream)
        solver.reset()
        if ev:
            ev[1].record(stream)
        solver.run()
        if ev:
            ev[2].record(stream)
        o = solver.observables()
        if ev:
            ev[3].record(stream)
        return o

    for _ in range(args.warmup):
        o = one_solve()
        if o.status != bte.OK:
            raise RuntimeError(f"solver status {o.status}")

    uuid = None
    try:
        uuid = str(torch.cuda.get_device_properties(dev).uuid)
    except Exception:
        pass
    clocks = ClockSampler(uuid)
    if world > 1:
        import torch.distributed as dist
        dist.barrier()
    torch.cuda.synchronize()
    clocks.start()
    evs = []
    for _ in range(args.steps):
        with torch.cuda.stream(stream):
            flush.fill_(1.0)
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(4)]
        o = one_solve(ev)
        evs.append(ev)
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    clk = clocks.stop()
    if o.status != bte.OK:
        raise RuntimeError(f"solver status {o.status}")
    step_ms = [e[0].elapsed_time(e[3]) for e in evs]
    run_ms = [e[1].elapsed_time(e[2]) for e in evs]
    total_ms = sum(step_ms)
    if world > 1:
        t = torch.tensor([total_ms, sum(run_ms)], device=dev, dtype=torch.float64)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        total_ms, run_total = t.tolist()
    else:
        run_total = sum(run_ms)
    value = world * cells * K * args.steps / (total_ms * 1e-3)

    # dominant kernel: average duration of one launch over the timed region
    # (run span / launches; includes inter-launch gaps): one or two steps, the
    # state read and written once.  On chip: reported per leap-frog step for
    # comparison
    avg_launch_s = run_total * 1e-3 / (args.steps * K) * (2 if kernel == "pair_kernel" else 1)
    alg_bytes = 8 * elem * cells
    hbm_peak, peak_kind = measured_peaks()
    achieved = alg_bytes / avg_launch_s / 1e9
    traffic = None if kernel != "pair_kernel" else ncu_traffic(f"{args.config}_{args.precision}")
    if state_bytes <= L2_BYTES * 3 // 4 and not on_chip:
        # the state stays in L2 between steps: L2 bandwidth is the roof
        bound, peak = "l2", measure_l2_gbs(dev)
        peak_source = "measured in this run: L2 copy of 2 x 24 MB (bench.py measure_l2_gbs)"
    else:
        bound, peak = "hbm", hbm_peak
        peak_source = peak_kind + " hbm_gbs"

    rate_unit = "GB/s"
    if kernel == "grid_kernel":
        # no memory traffic per step: the arithmetic is the roof (operations of
        # a cell-update as the kernel performs them)
        ops, rate_unit = (42, "T FP64 operations/s") if elem == 8 else (52, "T FP32 lane-ops/s")
        bound, achieved = "alu", cells / avg_launch_s * ops / 1e12
        peak, peak_source = (0.60, "measured FP64 rate") if elem == 8 else (
            40.27392, "152 SMs x 128 FP32 lanes x 2070 MHz (one lane operation per lane and clock; FMA counted once)")

    result_obs = o

    # end to end through the C ABI with host buffers: create (parameter and
    # table upload), run, observables (device -> host), destroy
    e2e = None
    if not args.no_e2e:
        pitch = bte.launch_shape(p, args.tile_m, args.chunk_n, args.vec)["pitch"]
        h2d = (p.n_max + 1) * elem + 2 * pitch * elem + 2 * 3 * (max(P, 1) + 2) * elem
        d2h = 4 * 8 + 2 * 8 + 4
        # a solve of several seconds needs no repetition for a stable figure
        e2e_steps = 1 if total_ms / args.steps > 5000 else max(1, min(args.steps, 3))
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for _ in range(e2e_steps):
            with bte.Solver(p, tile_m=args.tile_m, chunk_n=args.chunk_n,
                            graph_steps=args.graph_steps, vec=args.vec, resident=resident) as s2:
                s2.run()
                s2.observables()
        torch.cuda.synchronize()
        el = time.perf_counter() - t0
        if world > 1:
            t = torch.tensor([el], device=dev, dtype=torch.float64)
            dist.all_reduce(t, op=dist.ReduceOp.MAX)
            el = t.item()
        e2e = {"value": world * cells * K * e2e_steps / el, "unit": UNIT,
               "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(d2h)}

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        v, cores, n, el = oracle_sample(p.replace(precision=0), args.cpu_seconds)
        cpu = {"value": v, "unit": UNIT, "cores": cores, "kind": "oracle",
               "sample": f"{n} leap-frog steps of the {p.n_max + 1}x{p.m_points} grid "
                         f"(FP64 oracle, {el:.1f} s)"}

    solver.close()
    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": total_ms / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f64" if args.precision == "fp64" else "f32", "data": "synthetic",
            "config": {"workload": args.config + ": " + desc, "n_max": p.n_max,
                       "m_points": p.m_points, "steps_per_solve": K, "dt_eff": dt_eff,
                       "precision": "fp64" if args.precision == "fp64" else
                       "fp32 state, fp64 drive/reductions",
                       "l2": "flushed (256 MB write) before every timed step; the state "
                             f"({8 * elem * cells / 1e6:.0f} MB ping-pong) stays on chip within a solve "
                             "where it fits L2",
                       "parallelism": f"replicas x{world}",
                       "mode": {"on-chip": "on chip: the grid in one thread-block cluster's "
                                           "shared memory, one persistent launch per solve",
                                "on-chip-clusters": "on chip over several clusters: column blocks "
                                                    "in the shared memory of one cluster each, edge "
                                                    "columns exchanged through global memory, one "
                                                    "launch per 8192 steps",
                                "persistent": "persistent: one cooperative launch per 8192 steps, "
                                              "grid barrier between steps, state in L2",
                                "streamed": {"grid_kernel": "on chip, one block per SM: the grid in the "
                                                            "SMs' shared memory together, edges "
                                                            "exchanged through global memory",
                                             "pair_kernel": "two steps per launch, replayed from CUDA "
                                                            "graphs"}.get(
                                    kernel, "streamed: one fused step kernel launch per step, "
                                            "replayed from CUDA graphs")}[
                                    "streamed" if kernel == "grid_kernel" else mode],
                       "absorption": result_obs.absorption, "v_dc": result_obs.v_dc_avg,
                       "norm_max_abs_err": result_obs.norm_max_abs_err,
                       "fp32_vs_fp64": fp32_error(args, result_obs)},
            "roofline": {"bound": bound, "achieved": achieved, "peak": peak, "unit": rate_unit,
                         "frac": achieved / peak, "traffic": traffic,
                         "peak_source": peak_source,
                         "hbm_frac": alg_bytes / avg_launch_s / 1e9 / hbm_peak,
                         "kernel": kernel + (" (per step)" if on_chip or mode == "persistent" else ""),
                         "alg_bytes_per_launch": alg_bytes,
                         "avg_launch_us": avg_launch_s * 1e6},
            "cpu_baseline": cpu,
            "e2e": e2e,
            "gpu_launches": launches_per_solve * args.steps,
            "clocks": clk,
        }
        if world == 1 and not args.no_secondary:
            line["secondary"] = secondary(args)
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()
    return 0


def fp32_error(args, o):
    """Error of this FP32 full run against the FP64 full run of the same
    configuration (None for FP64 lines, shortened runs, or configurations
    without a recorded FP64 run)."""
    ref = FP64_FULL_RUN.get(args.config)
    if args.precision != "fp32" or args.periods or ref is None:
        return None
    return {"abs_err_absorption": abs(o.absorption - ref["absorption"]),
            "abs_err_v_dc": abs(o.v_dc_avg - ref["v_dc"]),
            "fp64_absorption": ref["absorption"], "fp64_v_dc": ref["v_dc"],
            "fp64_run": ref["how"]}


def secondary(args) -> dict:
    """The batched sweep and the surrogate measured once more in the same
    run, after the headline's timed region (context for the headline, each
    with its own roof): one timed pass over the 256-point stride sample of
    the 4096-point sweep (full 30-period runs), and 1M-point surrogate
    inference with training, held-out accuracy and the hybrid.  Not part of
    the headline's value or timed region."""
    import copy
    out = {}
    a = copy.copy(args)
    a.steps, a.warmup, a.no_e2e, a.no_cpu_baseline, a.periods = 1, 1, True, True, 0.0
    a.sweep_sample, a.single_sample, a.resident, a.tune = 256, 0, 0, False
    a.precision, a.tile_m, a.chunk_n, a.vec, a.graph_steps = "fp32", 0, 0, 0, 0
    a.sur_points, a.hybrid_sample, a.no_train = 1_000_000, 64, False
    keep = ("value", "unit", "ms_per_step", "roofline", "clocks")
    try:
        c4 = run_sweep(a, emit=False)
        out["c4"] = {k: c4.get(k) for k in keep}
        out["c4"]["config"] = {k: c4["config"].get(k) for k in
                               ("workload", "points_per_step", "sample", "cell_updates_per_s",
                                "tiers", "points_not_ok")}
    except Exception as e:  # reported, never fatal for the headline
        out["c4"] = {"error": repr(e)[:300]}
    try:
        a.steps = 3
        c5 = run_surrogate(a, emit=False)
        out["c5"] = {k: c5.get(k) for k in keep}
        out["c5"]["config"] = {k: c5["config"].get(k) for k in
                               ("workload", "points_per_step", "train_seconds", "heldout",
                                "hybrid", "fraction_to_solver")}
    except Exception as e:
        out["c5"] = {"error": repr(e)[:300]}
    return out


SWEEP_DESC = ("batched sweep: seeded uniform E_dc in [0,6], E_omega in [0.01,1], omega in [0.5,6], "
              "B in [0,6], mu in [0.5,10] (seed 1401); per-point n_max 20..200 and 201..2001 "
              "phi_y points by the grid rule; dt=1e-3, 30 periods, last 10 averaged")


def sweep_sample(args, world: int = 1):
    """The 4096-point sweep and the bounded sample of it one step solves:
    every (4096 / n)-th point (the points are i.i.d. draws, so a stride is
    an unbiased sample), n = sweep_sample x ranks (weak scaling: the work
    per GPU stays fixed)."""
    from paper_1401_6047_gb300 import workloads as W
    prec = W.FP64 if args.precision == "fp64" else W.FP32_MIXED
    if args.periods:
        # shortened runs (profiling): the grids and the mix of points stay the sweep's
        pts = W.sweep_points(4096, precision=prec, periods=args.periods,
                             avg_window=min(10.0, args.periods))
    else:
        pts = W.sweep_points(4096, precision=prec)
    n = max(1, min(4096, args.sweep_sample * world))
    stride = 4096 // n
    return pts[::stride][:n], stride


def sweep_launches(pts, max_batch, max_bytes, elem, tile, chunk, graph_len, tier):
    """Kernel launches of one bte_batch_run (same tiers and grouping rule as
    the library): on-chip points take 3 set-up launches each plus one
    persistent launch per cluster size in their batches; streamed points one
    launch per step of their batch plus graph counter updates."""
    from paper_1401_6047_gb300 import bte
    n = 0
    on = [(t, p) for t, p in zip(tier, pts) if t > 0]
    if on:
        # one batch per max_bytes of 4-array states, each with its own launches
        byt, sizes = 0, set()
        for t, p in on:
            _, P, _, _ = bte.time_grid(p)
            ntx = -(-p.m_points // tile)
            pitch = -(-(128 // elem + ntx * tile + 32 // elem) // 32) * 32
            sb = 4 * (p.n_max + 1) * pitch * elem + 6 * (P + 2) * elem + 4096
            if sizes and byt + sb > max_bytes:
                n += len(sizes)
                byt, sizes = 0, set()
            byt += sb
            sizes.add(int(t))
            n += 3
        n += len(sizes)
    info = []
    for t, p in zip(tier, pts):
        if t > 0:
            continue
        _, P, K, _ = bte.time_grid(p)
        info.append((K, P, p))
    info.sort(key=lambda t: -t[0])
    i = 0
    while i < len(info):
        j, byt = i, 0
        while j < len(info) and j - i < max_batch:
            K, P, p = info[j]
            ntx = -(-p.m_points // tile)
            pitch = -(-(128 // elem + ntx * tile + 32 // elem) // 32) * 32
            sb = 8 * (p.n_max + 1) * pitch * elem + 6 * (P + 2) * elem + 4096
            if j > i and byt + sb > max_bytes:
                break
            byt += sb
            j += 1
        Kmax = info[i][0]
        L = min(graph_len, Kmax)
        full = Kmax // L if L >= 2 else 0
        left = Kmax - full * L
        n += 3 * (j - i) + Kmax + full + (1 if left else 0)
        i = j
    return n


def run_sweep(args, emit: bool = True):
    import torch
    world, rank, local = dist_setup()
    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    dev = torch.device("cuda", torch.cuda.current_device())
    from paper_1401_6047_gb300 import bte

    allpts, stride = sweep_sample(args, world)
    # weak scaling: the sample grows with the ranks; rank r solves its share
    from paper_1401_6047_gb300 import shard
    cost = [p.cells * bte.time_grid(p)[2] for p in allpts]
    pts = [allpts[i] for i in shard.split(len(allpts), rank, world, cost)]
    elem = 8 if args.precision == "fp64" else 4
    vec = args.vec or (2 if elem == 8 else 4)
    tile = args.tile_m or 64 * vec
    chunk = args.chunk_n or 16
    max_batch = args.max_batch or 1024
    max_bytes = args.max_batch_bytes or (4 << 30)
    cu = 0
    for p in pts:
        cu += p.cells * bte.time_grid(p)[2]
    stream = torch.cuda.Stream(device=dev)
    kw = dict(tile_m=tile, chunk_n=chunk, vec=vec, graph_steps=args.graph_steps,
              max_batch=max_batch, max_batch_bytes=max_bytes, stream=stream.cuda_stream,
              resident=args.resident, resident_smem=args.resident_smem)
    tuned = None
    if args.tune:
        # the library's autotuner on the same points (shortened runs), before timing
        t0 = time.perf_counter()
        best, secs = bte.batch_tune(pts, sample=16, steps=2000,
                                    **{k: v for k, v in kw.items() if k != "stream"})
        tuned = {"options": best, "seconds": time.perf_counter() - t0,
                 "candidate_seconds": [None if s > 1e299 else s for s in secs.tolist()]}
        kw.update(best)
        tile, chunk, vec = kw["tile_m"] or tile, kw["chunk_n"] or chunk, kw["vec"] or vec
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    for _ in range(args.warmup):
        res = bte.batch_run(pts, **kw)
    uuid = None
    try:
        uuid = str(torch.cuda.get_device_properties(dev).uuid)
    except Exception:
        pass
    clocks = ClockSampler(uuid)
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    clocks.start()
    evs = []
    for _ in range(args.steps):
        with torch.cuda.stream(stream):
            flush.fill_(1.0)
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record(stream)
        res = bte.batch_run(pts, **kw)
        e[1].record(stream)
        evs.append(e)
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    clk = clocks.stop()
    total_ms = sum(e[0].elapsed_time(e[1]) for e in evs)
    if world > 1:
        t = torch.tensor([total_ms], device=dev, dtype=torch.float64)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        total_ms = t.item()
    secs = total_ms * 1e-3
    value = len(allpts) * args.steps / secs
    bad = sum(1 for o in res if o.status != bte.OK)
    peak, peak_kind = measured_peaks()
    achieved = 8 * elem * cu * args.steps / (secs / 1 if world == 1 else secs) / 1e9
    graph_len = args.graph_steps or 1024
    tier = bte.batch_plan(pts, **{k: v for k, v in kw.items() if k != "stream"})
    launches = sweep_launches(pts, max_batch, max_bytes, elem, tile, chunk, graph_len, tier)
    cu_on = sum(p.cells * bte.time_grid(p)[2] for t, p in zip(tier, pts) if t > 0)

    # end to end: host parameter array in, host results out, through the C ABI
    # (bte_batch_run allocates, uploads tables, runs, reads back and frees)
    e2e = None
    if not args.no_e2e:
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        bte.batch_run(pts, **{k: v for k, v in kw.items() if k != "stream"})
        torch.cuda.synchronize()
        el = time.perf_counter() - t0
        if world > 1:
            t = torch.tensor([el], device=dev, dtype=torch.float64)
            dist.all_reduce(t, op=dist.ReduceOp.MAX)
            el = t.item()
        e2e = {"value": len(allpts) / el, "unit": "points/s",
               "h2d_bytes_per_step": len(pts) * 112, "d2h_bytes_per_step": len(pts) * 96}

    # the plain single-instance GPU solver on a few of the same points
    single = None
    if rank == 0 and args.single_sample > 0:
        sub = pts[:: max(1, len(pts) // args.single_sample)][: args.single_sample]
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for p in sub:
            bte.solve(p, stream=stream.cuda_stream)
        torch.cuda.synchronize()
        el = time.perf_counter() - t0
        cu_sub = sum(p.cells * bte.time_grid(p)[2] for p in sub)
        # scale to the sample's mix by cell-updates
        single = {"points_per_s": len(sub) / el * (cu_sub / len(sub)) / (cu / len(pts)),
                  "cell_updates_per_s": cu_sub / el, "points": len(sub),
                  "note": "bte_solve one point after another on the same stream; points/s "
                          "scaled to the sample's mean cell-updates per point"}

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        p0 = pts[0].replace(precision=0)
        v, cores, n, el = oracle_sample(p0, args.cpu_seconds)
        cpu = {"value": v / (cu / len(pts)), "unit": "points/s", "cores": cores, "kind": "oracle",
               "sample": f"{n} steps of sweep point 0 ({p0.n_max + 1}x{p0.m_points}, FP64 "
                         f"oracle, {el:.1f} s) = {v:.3e} cell-updates/s, divided by the "
                         f"sample's mean {cu / len(pts):.3e} cell-updates per point"}
    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": "points/s", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": total_ms / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f64" if elem == 8 else "f32", "data": "synthetic",
            "config": {"workload": "c4: " + SWEEP_DESC, "points_per_step": len(allpts),
                       "sample": f"every {stride}th of the 4096 points",
                       "cell_updates_per_step": cu * world, "cell_updates_per_s": cu * world * args.steps / secs,
                       "precision": "fp64" if elem == 8 else "fp32 state, fp64 drive/reductions",
                       "tile_m": tile, "chunk_n": chunk, "vec": vec, "max_batch": max_batch,
                       "tiers": {str(int(t)): int((tier == t).sum()) for t in sorted(set(tier.tolist()))},
                       "max_batch_bytes": max_bytes, "points_not_ok": bad,
                       "l2": "flushed (256 MB write) before every timed step",
                       "parallelism": f"points split over {world} rank(s)"},
            "roofline": sweep_roofline(cu * world * args.steps / secs, achieved, peak, peak_kind,
                                       cu_on / cu if cu else 0.0, elem, clk),
            "cpu_baseline": cpu, "single_instance_gpu": single, "e2e": e2e, "tuned": tuned,
            "gpu_launches": launches * args.steps, "clocks": clk,
        }
        if not emit:
            return line
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()
    return 0


# FP32 lane operations (multiply, add, fused multiply-add) of one cell-update,
# both grids: 24 per cell of a half-step in the Crank-Nicolson update and 2
# for the phi_y differences of the row it contributes (the reciprocal of the
# denominator runs on the special-function unit and is not counted)
FP32_OPS_PER_CELL_UPDATE = 52


def sweep_roofline(cell_updates_per_s, hbm_achieved, hbm_peak, peak_kind, on_chip_share, elem, clk):
    """Roof of the batched sweep.  When the on-chip tier carries (nearly)
    every cell-update the state never leaves shared memory, so the bound is
    the FP32 arithmetic: 152 SMs x 128 FP32 lanes x the SM clock (the
    maximum, 2070 MHz, when no clock sample is at hand) against
    FP32_OPS_PER_CELL_UPDATE lane operations per cell-update.  Otherwise
    the HBM roof of the streamed tier with 32 / 64 B per cell-update."""
    if elem == 4 and on_chip_share >= 0.99:
        mhz = (clk or {}).get("sm_max_mhz") or 2070.0
        peak = 152 * 128 * mhz * 1e6 / 1e12  # Tops/s
        achieved = cell_updates_per_s * FP32_OPS_PER_CELL_UPDATE / 1e12
        return {"bound": "alu", "achieved": achieved, "peak": peak,
                "unit": "T FP32 lane-ops/s", "frac": achieved / peak, "traffic": None,
                "peak_source": f"152 SMs x 128 FP32 lanes x {mhz:.0f} MHz (one lane operation per "
                               f"lane and clock; FMA counted once)",
                "ops_per_cell_update": FP32_OPS_PER_CELL_UPDATE,
                "kernel": "resident_kernel (on-chip tier)",
                "on_chip_share_of_cell_updates": on_chip_share,
                "hbm_equivalent": {"achieved_gbs": hbm_achieved, "peak_gbs": hbm_peak,
                                   "note": "algorithmic bytes of the streamed form, for comparison"}}
    return {"bound": "hbm", "achieved": hbm_achieved, "peak": hbm_peak, "unit": "GB/s",
            "frac": hbm_achieved / hbm_peak, "traffic": None,
            "peak_source": peak_kind + " hbm_gbs",
            "kernel": "resident_kernel (on-chip tier) + fused_step_kernel (streamed tier)",
            "on_chip_share_of_cell_updates": on_chip_share,
            "note": "algorithmic bytes (32 B FP32 / 64 B FP64 per cell-update) over the whole "
                    "batch solve"}


def run_sweep_reference(args):
    world, rank, _ = dist_setup()
    if rank != 0:
        return 0
    import oracle
    from paper_1401_6047_gb300 import bte
    oracle.build()
    pts, stride = sweep_sample(args)
    mean_cu = sum(p.cells * bte.time_grid(p)[2] for p in pts) / len(pts)
    per_step = max(1.0, 60.0 / max(1, args.steps + args.warmup))
    for i in range(args.warmup):
        oracle_sample(pts[i % len(pts)].replace(precision=0), min(per_step, 5.0))
    cus, secs, cores = 0.0, 0.0, 0
    for i in range(args.steps):
        p = pts[(7 * i) % len(pts)].replace(precision=0)
        v, cores, n, el = oracle_sample(p, per_step)
        cus += p.cells * n
        secs += el
    value = cus / secs / mean_cu
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": "points/s",
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": 1e3 * secs / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": "c4: " + SWEEP_DESC, "points_per_step": len(pts),
                   "precision": "fp64 (oracle)"},
        "cpu_baseline": {"value": value, "unit": "points/s", "cores": cores, "kind": "oracle",
                         "sample": f"{args.steps} bounded runs of sweep points; cell-updates/s "
                                   f"divided by the mean {mean_cu:.3e} cell-updates per point"},
        "e2e": {"value": value, "unit": "points/s", "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


SUR_DESC = ("learned surrogate: 8-member ensemble of MLP 5-256-256-256-2 (SiLU), BF16 tensor-core "
            "layers with FP32 accumulation, trained on 200,000 sweep-box points (seed 6047) solved "
            "by the batched solver, judged on 10,240 held-out points (seed 2015); inference on 1M "
            "seeded points (seed 2014) of the same box, solver fallback where the ensemble std "
            "exceeds 1e-3")


def sur_flops_per_point(members=8, H=256):
    """Multiply-adds x 2 of one forward pass of every member."""
    return members * 2 * (5 * H + 2 * H * H + 2 * H)


def run_surrogate(args, emit: bool = True):
    import numpy as np
    import torch

    world, rank, local = dist_setup()
    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    dev = torch.device("cuda", torch.cuda.current_device())
    from paper_1401_6047_gb300 import bte
    from paper_1401_6047_gb300 import surrogate as S
    from paper_1401_6047_gb300 import surrogate_data as D
    from paper_1401_6047_gb300 import workloads as W

    x_tr, y_tr = D.load("train")
    x_ho, y_ho = D.load("heldout")
    stream = torch.cuda.Stream(device=dev)
    sur = S.Surrogate(y_tr.mean(axis=0), y_tr.std(axis=0), members=8, batch_capacity=65536,
                      stream=stream.cuda_stream)
    sur.set_params(S.init_params(8, seed=0))
    t0 = time.perf_counter()
    # --no-train (profiling only): inference cost does not depend on the weights
    hist = [float("nan")] if args.no_train else sur.fit(x_tr, y_tr, **D.TRAINING)
    train_s = time.perf_counter() - t0

    n = args.sur_points
    xs = W.sweep_matrix(n * world, W.SURROGATE_INFER_SEED)[rank * n:(rank + 1) * n]
    xd = torch.from_numpy(xs.astype(np.float32)).to(dev)
    md = torch.empty((n, 2), device=dev)
    sd = torch.empty((n, 2), device=dev)
    kd = torch.empty(n, dtype=torch.uint8, device=dev)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)

    def step():
        sur.predict_device(xd.data_ptr(), n, md.data_ptr(), sd.data_ptr(), kd.data_ptr(), 1e-3)

    for _ in range(args.warmup):
        step()
    uuid = None
    try:
        uuid = str(torch.cuda.get_device_properties(dev).uuid)
    except Exception:
        pass
    clocks = ClockSampler(uuid)
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    clocks.start()
    evs = []
    for _ in range(args.steps):
        with torch.cuda.stream(stream):
            flush.fill_(1.0)
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        e[0].record(stream)
        step()
        e[1].record(stream)
        evs.append(e)
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    clk = clocks.stop()
    total_ms = sum(a.elapsed_time(b) for a, b in evs)
    if world > 1:
        t = torch.tensor([total_ms], device=dev, dtype=torch.float64)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        total_ms = t.item()
    secs = total_ms * 1e-3
    value = world * n * args.steps / secs
    frac_solver = float(kd.float().mean().item())
    flops = sur_flops_per_point() * n
    tflops = flops * args.steps / secs / 1e12
    peaks = {}
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            peaks = json.load(f)
    except Exception:
        pass
    peak = float(peaks.get("bf16_tflops", 1900.0))

    # end to end: host inputs in, host mean / std / mask out, through the
    # public host-array call, page-locked host buffers (the library overlaps
    # each chunk's copies with the next chunk's inference)
    e2e = None
    if not args.no_e2e:
        xp = torch.empty((n, 5), dtype=torch.float32, pin_memory=True)
        xp.numpy()[:] = np.asarray(xs, dtype=np.float32)
        outs = (torch.empty((n, 2), dtype=torch.float32, pin_memory=True).numpy(),
                torch.empty((n, 2), dtype=torch.float32, pin_memory=True).numpy(),
                torch.empty(n, dtype=torch.uint8, pin_memory=True).numpy())
        sur.predict(xp.numpy(), threshold=1e-3, out=outs)  # warm-up (creates the copy streams)
        e2e_steps = max(1, min(args.steps, 3))
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for _ in range(e2e_steps):
            sur.predict(xp.numpy(), threshold=1e-3, out=outs)
        el = (time.perf_counter() - t0) / e2e_steps
        e2e = {"value": world * n / el, "unit": "points/s", "h2d_bytes_per_step": int(n * 20),
               "d2h_bytes_per_step": int(n * 17), "host_buffers": "page-locked"}

    # accuracy on held-out solver results, and the hybrid against the solver alone
    mean, std, mask = sur.predict(x_ho, threshold=1e-3)
    err = np.abs(mean - y_ho).max(axis=1)
    acc = ~mask
    hybrid = None
    accuracy = None
    if rank == 0 and args.hybrid_sample > 0:
        sample = x_ho[:: max(1, len(x_ho) // args.hybrid_sample)][: args.hybrid_sample]
        pts = [S.protocol(xi) for xi in sample]
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        bte.batch_run(pts)
        t_solver = time.perf_counter() - t0
        t0 = time.perf_counter()
        yh, solved, _ = sur.hybrid(sample, threshold=1e-3)
        t_hybrid = time.perf_counter() - t0
        solver_rate = len(sample) / t_solver
        hybrid = {"points": len(sample), "threshold": 1e-3,
                  "hybrid_points_per_s": len(sample) / t_hybrid,
                  "solver_only_points_per_s": solver_rate,
                  "fraction_solved": float(solved.mean())}
        accuracy = sur_accuracy_table(mean, std, y_ho, value, solver_rate)
    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        from oracle import mlp
        P = sur.get_params().astype(np.float64)
        lo, hi = S.box_bounds()
        m0 = 2048
        t0 = time.perf_counter()
        cnt = 0
        while time.perf_counter() - t0 < args.cpu_seconds:
            mlp.ensemble(list(P), xs[cnt % (n - m0):cnt % (n - m0) + m0], lo, hi,
                         y_tr.mean(axis=0), y_tr.std(axis=0))
            cnt += m0
        el = time.perf_counter() - t0
        cpu = {"value": cnt / el, "unit": "points/s", "cores": os.cpu_count(), "kind": "oracle",
               "sample": f"{cnt} points through the FP64 numpy ensemble ({el:.1f} s; numpy's "
                         f"BLAS threads)"}
    sur.close()
    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": "points/s", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": total_ms / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16",
            "data": "synthetic",
            "config": {"workload": "c5: " + SUR_DESC, "points_per_step": n * world,
                       "train_seconds": train_s, "train_final_loss": hist[-1],
                       "fraction_to_solver": frac_solver,
                       "heldout": {"points": int(len(x_ho)), "accepted": float(acc.mean()),
                                   "err_p50_accepted": float(np.median(err[acc])) if acc.any() else None,
                                   "err_p99_accepted": float(np.quantile(err[acc], 0.99)) if acc.any() else None,
                                   "err_max_accepted": float(err[acc].max()) if acc.any() else None,
                                   "err_p50_all": float(np.median(err))},
                       "hybrid": hybrid, "accuracy": accuracy,
                       "l2": "flushed (256 MB write) before every timed step; inputs 20 MB"},
            "roofline": {"bound": "tensor", "achieved": tflops, "peak": peak, "unit": "TFLOP/s",
                         "frac": tflops / peak, "traffic": None,
                         "peak_source": "measured bf16_tflops (cuBLAS burst)",
                         "kernel": "infer_tc_kernel (tcgen05; plus the ensemble mean/std kernel, "
                                   "one of each per 65,536-point chunk)",
                         "flops_per_point": sur_flops_per_point()},
            "cpu_baseline": cpu, "e2e": e2e,
            "gpu_launches": (2 * (-(-n // 65536)) + 1) * args.steps, "clocks": clk,
        }
        if not emit:
            return line
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()
    return 0


def sur_accuracy_table(mean, std, y_ref, infer_rate, solver_rate):
    """Each form of the surrogate at the accuracy it reaches on the held-out
    solver results: the surrogate alone, the hybrid (solver wherever the
    ensemble std exceeds the threshold) at 1e-3 and 1e-4, and the hybrid at
    the largest threshold whose accepted held-out points all lie within the
    metric's 1e-5 absolute bar.  Points/s of a hybrid = points / (inference
    time + fallback fraction x points / solver points/s), from the measured
    inference and solver rates; the solver's own error is that of the FP32
    batched solver (1e-5 absolute against the FP64 oracle by the parity
    tests)."""
    import numpy as np
    err = np.abs(mean - y_ref).max(axis=1)
    spread = std.max(axis=1)

    def row(thr):
        acc = spread <= thr
        f = 1.0 - float(acc.mean())
        rate = 1.0 / (1.0 / infer_rate + f / solver_rate)
        return {"threshold": thr, "fraction_to_solver": f,
                "max_abs_err": float(err[acc].max()) if acc.any() else 0.0,
                "p99_abs_err": float(np.quantile(err[acc], 0.99)) if acc.any() else 0.0,
                "points_per_s": rate}
    out = {"surrogate_only": row(float("inf")), "hybrid_1e-3": row(1e-3), "hybrid_1e-4": row(1e-4)}
    # the largest threshold meeting the 1e-5 bar on every accepted point
    order = np.argsort(spread)
    bad = np.cumsum(err[order] > 1e-5)
    ok_n = int(np.searchsorted(bad, 1))  # points before the first one above the bar
    thr = float(spread[order[ok_n - 1]]) if ok_n > 0 else 0.0
    r = row(thr)
    r["note"] = "largest threshold whose accepted held-out points are all within 1e-5 absolute"
    out["hybrid_at_1e-5"] = r
    out["solver_only"] = {"points_per_s": solver_rate, "max_abs_err": 1e-5,
                          "note": "FP32 batched solver; error bound from the GPU-vs-oracle tests"}
    return out


def run_surrogate_reference(args):
    world, rank, _ = dist_setup()
    if rank != 0:
        return 0
    import numpy as np
    from oracle import mlp
    from paper_1401_6047_gb300 import surrogate as S
    from paper_1401_6047_gb300 import surrogate_data as D
    from paper_1401_6047_gb300 import workloads as W
    x_tr, y_tr = D.load("train")
    P = [mlp.init_member(m) for m in range(8)]
    lo, hi = S.box_bounds()
    xs = W.sweep_matrix(65536, W.SURROGATE_INFER_SEED)
    per_step = max(1.0, 60.0 / max(1, args.steps + args.warmup))
    m0 = 2048

    def sample(limit):
        t0 = time.perf_counter()
        cnt = 0
        while time.perf_counter() - t0 < limit:
            mlp.ensemble(P, xs[cnt % 60000:cnt % 60000 + m0], lo, hi, y_tr.mean(axis=0),
                         y_tr.std(axis=0))
            cnt += m0
        return cnt, time.perf_counter() - t0

    for _ in range(args.warmup):
        sample(min(per_step, 3.0))
    cnt, el = 0, 0.0
    for _ in range(args.steps):
        c, e = sample(per_step)
        cnt += c
        el += e
    value = cnt / el
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": "points/s",
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": 1e3 * el / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": "c5: " + SUR_DESC, "precision": "fp64 (oracle)"},
        "cpu_baseline": {"value": value, "unit": "points/s", "cores": os.cpu_count(),
                         "kind": "oracle",
                         "sample": f"{cnt} points through the FP64 numpy ensemble"},
        "e2e": {"value": value, "unit": "points/s", "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


def main():
    ap = argparse.ArgumentParser(description=__doc__.split("\n")[0])
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--config", default="c3", choices=["c1", "c2", "c3", "table1", "c4", "c5"])
    ap.add_argument("--precision", default="fp32", choices=["fp32", "fp64"])
    ap.add_argument("--tile-m", dest="tile_m", type=int, default=0)
    ap.add_argument("--chunk-n", dest="chunk_n", type=int, default=0)
    ap.add_argument("--graph-steps", dest="graph_steps", type=int, default=0)
    ap.add_argument("--vec", type=int, default=0)
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--cpu-seconds", type=float, default=15.0)
    ap.add_argument("--periods", type=float, default=0.0,
                    help="shorter run (drive periods) for profiling; 0 = the workload's")
    ap.add_argument("--sweep-sample", dest="sweep_sample", type=int, default=256,
                    help="c4: points of the 4096-point sweep solved per step")
    ap.add_argument("--max-batch", dest="max_batch", type=int, default=0)
    ap.add_argument("--tune", action="store_true",
                    help="c4: pick the batched-run options with the library's autotuner first")
    ap.add_argument("--resident", type=int, default=0,
                    help="c4: 0 on chip where a point fits, 1 never, 2 only")
    ap.add_argument("--resident-smem", dest="resident_smem", type=int, default=0,
                    help="c4: shared memory per CTA for on-chip points (bytes)")
    ap.add_argument("--max-batch-bytes", dest="max_batch_bytes", type=int, default=0)
    ap.add_argument("--mode", default="auto",
                    choices=["auto", "streamed", "persistent", "on-chip", "on-chip-clusters"],
                    help="single-instance mode (auto: streamed, one launch per step)")
    ap.add_argument("--on-chip", dest="on_chip", action="store_true",
                    help="single-instance configs: keep the grid in one cluster's shared memory")
    ap.add_argument("--single-sample", dest="single_sample", type=int, default=8,
                    help="c4: points solved one by one for the single-instance comparison")
    ap.add_argument("--sur-points", dest="sur_points", type=int, default=1_000_000,
                    help="c5: points per inference step")
    ap.add_argument("--no-train", dest="no_train", action="store_true",
                    help="c5: skip training (profiling the inference kernels only)")
    ap.add_argument("--hybrid-sample", dest="hybrid_sample", type=int, default=256,
                    help="c5: held-out points timed through the surrogate with solver fallback")
    ap.add_argument("--no-secondary", dest="no_secondary", action="store_true",
                    help="single-instance configs: skip the sweep and surrogate measured after "
                         "the headline")
    args = ap.parse_args()
    if args.warmup < 3:
        print("warning: fewer than 3 warm-up steps", file=sys.stderr)
    if args.config == "c5":
        return run_surrogate_reference(args) if args.impl == "reference" else run_surrogate(args)
    if args.config == "c4":
        return run_sweep_reference(args) if args.impl == "reference" else run_sweep(args)
    if args.impl == "reference":
        return run_reference(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
