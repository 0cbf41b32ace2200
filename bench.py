"""Throughput of the axisymmetric Shan-Chen LBM step on GB300 (MLUPS and HBM roofline).

Workload: the batched sweep of 64 independent drops (R ~ U[10, 60], grid 4R x 2R,
G ~ U[-5.5, -4.6], tau ~ U[0.6, 1.2], l = 2 amplitude ~ U[0, 0.08] on half of
them, seeds 1234 + k), populations stored in FP32 with FP32 arithmetic (the form
whose density stays within 1e-4 of the FP64 form; the BF16 and FP16 forms are
reported beside it with their errors), all instances in one kernel launch per
timestep.

One bench step = one timestep of every site of every instance.  The state
(~58 MB) fits in L2, so L2 is flushed (a 256 MB write) before every timed step
and each step is timed alone with CUDA events on the launching stream: the
figure is the HBM-fed rate, a lower bound on a run that stays L2-resident.  The
same steps replayed back to back from a captured CUDA graph are reported beside it.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]

Under torchrun (N > 1) every rank runs its own 64-instance batch (seeds offset by
64 x rank): independent problems, no collective on the data path (weak scaling).
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from paper_1310_1871_gb300 import inputs as I  # noqa: E402

METRIC = "MLUPS & % of HBM roofline, mixed-precision/batched vs plain FP64 at same error"
UNIT = "MLUPS"
STORAGE = "f32"
BYTES_PER_LU = {"f64": 18 * 8 + 2 * 8, "f32": 18 * 4 + 2 * 4, "f16": 18 * 2 + 2 * 4, "bf16": 18 * 2 + 2 * 4}
WORKLOAD = ("batched sweep: 64 axisymmetric drops, R~U[10,60], grid 4R x 2R, G~U[-5.5,-4.6], "
            "tau~U[0.6,1.2], a2~U[0,0.08] on odd instances, seeds 1234+k")


def config(sites, storage=STORAGE, tile=None, schedule=None):
    return {"workload": WORKLOAD, "instances": 64, "sites_per_step": int(sites),
            "storage": (f"{storage}, f_i - W_i*rho(psi) (site density recovered from psi)"
                        if storage in ("f16", "bf16") else
                        f"{storage} populations (unshifted), max rel rho error vs FP64 <= 1e-4"),
            "arithmetic": "f64" if storage == "f64" else "f32",
            "schedule": schedule, "tile": list(tile) if tile else None,
            "l2": "flushed before every timed step (256 MB write); state < L2",
            "launch": "every tile of all 64 instances in one launch per kernel per timestep"}


def profiled_traffic(kernel_src, kernel):
    """DRAM bytes per launch of a step kernel from the committed ncu summary, or None
    when that kernel was not captured or its source changed since."""
    p = os.path.join(ROOT, "profiles", "step_kernel_traffic.json")
    if not os.path.exists(p):
        return None
    d = json.load(open(p))
    sha = hashlib.sha256(open(kernel_src, "rb").read()).hexdigest()
    for part in (d, d.get("strips", {})):  # the pair schedule's tiles, and its strips
        if part.get("source_sha256") == sha and kernel in part.get("kernels", {}):
            return part["kernels"][kernel].get("dram_bytes_per_launch")
    return None


def autotune_summary(tuned):
    """The autotuner's five fastest candidates (schedule, tile, MLUPS on back-to-back steps)."""
    if not tuned:
        return None
    c = sorted(tuned["candidates"], key=lambda x: x["ms_per_step"])
    return {"chosen": [tuned["schedule"], tuned["tile"]], "cached": tuned.get("cached"),
            "candidates": len(c),
            "top": [[x["schedule"], x["tile"], round(x["mlups"], 1)] for x in c[:5]]}


def peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


class ClockSampler:
    """nvidia-smi samples of SM clock and throttle reasons while the timed loop runs."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.lines = []

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "50"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except OSError:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def __exit__(self, *a):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
            self.t.join(timeout=2)

    def summary(self):
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [x.strip() for x in ln.split(",")]
            if len(parts) < 7:
                continue
            try:
                sm.append(float(parts[0]))
                mx = float(parts[1])
            except ValueError:
                continue
            for n, v in zip(names, parts[3:7]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": mx,
                "reasons": sorted(reasons), "samples": len(sm)}


def rank_seed0(rank):
    """First seed of a rank's 64-instance batch: ranks run disjoint, independent batches."""
    return 1234 + 64 * rank


def max_over_ranks(value, world, device="cpu"):
    """The largest per-rank value (the whole job is as slow as its slowest rank)."""
    if world <= 1:
        return float(value)
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(value)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def sum_over_ranks(value, world, device="cpu"):
    """The sum of a per-rank value over all ranks."""
    if world <= 1:
        return float(value)
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(value)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.SUM)
    return float(t.item())


def job_mlups(job_sites, steps, max_ms):
    """Whole-job lattice updates per second (millions): the sites of all ranks (each
    rank its own batch), over the slowest rank's time."""
    return job_sites * steps / (max_ms * 1e-3) / 1e6


def parse_launch(text):
    """'auto' or 'SCHEDULE:TZxTR' (e.g. pair:32x16) -> (tile, schedule) for amlbm.Batch."""
    if text == "auto":
        return "auto", "auto"
    sched, tile = text.split(":")
    tz, tr = (int(v) for v in tile.lower().split("x"))
    return (tz, tr), sched


def build_batch(storage, rank, tile="auto", graph_chunk=0, stream=None, schedule="auto"):
    from paper_1310_1871_gb300 import amlbm
    inst = I.batch_sweep(64, seed0=rank_seed0(rank))
    specs = [amlbm.InstanceSpec(x.Nz, x.Nr, x.tau, x.G) for x in inst]
    b = amlbm.Batch(specs, storage=storage, tile=tile, graph_chunk=graph_chunk, stream=stream,
                    schedule=schedule)
    for k, x in enumerate(inst):
        b.init_fields(k, *x.make_fields())
    return b, inst


def time_steps(torch, b, steps, warmup, flush, stream):
    """Per-step CUDA-event times (ms) of `steps` timesteps, L2 flushed before each."""
    for _ in range(warmup):
        flush.add_(1)
        b.step(1)
    torch.cuda.synchronize()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
    for s in range(steps):
        flush.add_(1)  # 256 MB read-modify-write on the same stream evicts the state from L2
        ev[s][0].record(stream)
        b.step(1)
        ev[s][1].record(stream)
    torch.cuda.synchronize()
    return [a.elapsed_time(c) for a, c in ev]


def run_gpu(args):
    import torch
    import torch.distributed as dist

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    torch.cuda.set_device(local)
    stream = torch.cuda.Stream()
    flush = torch.empty(256 * 2 ** 20 // 4, dtype=torch.float32, device="cuda")
    with torch.cuda.stream(stream):
        tile0, sched0 = parse_launch(args.launch)
        b, inst = build_batch(STORAGE, rank, tile=tile0, schedule=sched0, stream=stream)
        sites = b.sites
        sched, tile, lps = b.schedule, b.tile, b.launches_per_step
        tuned = b.tuned
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()
        with ClockSampler(local) as clk:
            t0 = time.perf_counter()
            times = time_steps(torch, b, args.steps, args.warmup, flush, stream)
            wall = time.perf_counter() - t0
        total_ms = max_over_ranks(float(sum(times)), world, "cuda")
        if world > 1:
            dist.barrier()
        job_sites = sum_over_ranks(sites, world, "cuda")
        mlups = job_mlups(job_sites, args.steps, total_ms)
        avg_ms = total_ms / args.steps
        # the timed steps split into five consecutive chunks: median and spread of
        # the chunks' MLUPS (one run, not five)
        runs = [sites * len(c) / (sum(c) * 1e-3) / 1e6 for c in np.array_split(np.array(times), 5) if len(c)]
        five = {"median_mlups": round(float(np.median(runs)), 1), "min_mlups": round(min(runs), 1),
                "max_mlups": round(max(runs), 1)}
        hbm, kind = peaks()
        achieved = BYTES_PER_LU[STORAGE] * sites / (avg_ms * 1e-3) / 1e9
        b.close()
        graph = graph_back_to_back(torch, rank, stream, max(20, min(args.steps, 2000)), tile0, sched0)
        b, inst = build_batch(STORAGE, rank, tile=tile0, schedule=sched0, stream=stream)

        # end to end through the public C ABI: every step uploads every instance's
        # fields from pinned host memory (one copy per field array for the whole
        # batch), runs one timestep, and reads every instance's diagnostics (FP64
        # reductions) back to the host
        # The FP32 form computes in FP32 and rounds its inputs to FP32 first, so
        # its fields go up as FP32 (amlbm_batch_init_all_f32, the same state); the
        # FP64 fields are timed as well (e2e_fp64_inputs).
        e2e_steps = max(3, min(args.steps, 50))
        cols = [np.concatenate([np.ravel(x.make_fields()[q]) for x in inst]) for q in range(3)]
        params = np.array([[x.zc, x.R, x.rho_l, x.rho_v] for x in inst], dtype=np.float64)
        d2h = 64 * 16 * 8

        def e2e_run(dtype):
            pinned = [torch.from_numpy(c.astype(dtype)).pin_memory() for c in cols]
            host = [t.numpy() for t in pinned]
            b.init_all(*host)
            b.step(1)
            b.diagnostics_all(params, check=False, as_array=True)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            for _ in range(e2e_steps):
                b.init_all(*host)
                b.step(1)
                b.diagnostics_all(params, check=False, as_array=True)
            torch.cuda.synchronize()
            e2e_s = time.perf_counter() - t0
            return (job_mlups(job_sites, e2e_steps, max_over_ranks(e2e_s, world, "cuda") * 1e3),
                    sum(a.nbytes for a in host))

        e2e_val, h2d = e2e_run(np.float32 if STORAGE != "f64" else np.float64)
        e2e64_val, h2d64 = e2e_run(np.float64)
        b.close()

        # the same workload in the other storage forms (plain FP64 is the
        # parity form; FP32 the unshifted single-precision form)
        compare = {}
        adjoint = None
        scaled = None
        precision = None
        if rank == 0 and not args.no_compare:
            # the other storage forms on the same flushed-L2 timing (plain FP64 is the
            # parity form; the W_i s-shifted BF16 form misses the 1e-4 error target,
            # see precision_vs_f64)
            for st in ("f64", "bf16"):
                bb, _ = build_batch(st, rank, stream=stream)
                tt = time_steps(torch, bb, min(args.steps, 200), 3, flush, stream)
                compare[st] = {"mlups": round(bb.sites * len(tt) / (sum(tt) * 1e-3) / 1e6, 1),
                               "schedule": bb.schedule, "tile": list(bb.tile)}
                bb.close()
            compare["bf16"]["meets_1e-4"] = False
            compare[STORAGE] = {"mlups": round(mlups / world, 1), "schedule": sched, "tile": list(tile),
                                "meets_1e-4": True}
            compare["f32_over_f64_at_same_error"] = round(compare[STORAGE]["mlups"] / compare["f64"]["mlups"], 2)
            adjoint = adjoint_cost(torch)
            scaled = scaled_cases(torch, tile, sched)
            precision = precision_vs_f64(torch)

    kname, ksrc = kernel_name(STORAGE, sched, tile)
    traffic = profiled_traffic(ksrc, kname)
    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu:
        cpu = cpu_baseline(seconds=args.cpu_seconds)
    if rank == 0:
        line = {
            "metric": METRIC, "value": round(mlups, 1), "unit": UNIT, "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(avg_ms, 6),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic", "config": dict(config(sites, tile=tile, schedule=sched),
                                                autotune=autotune_summary(tuned)),
            "roofline": {"bound": "hbm", "achieved": round(achieved, 1), "peak": hbm, "unit": "GB/s",
                         "frac": round(achieved / hbm, 4),
                         "traffic": (round(traffic) if traffic else None),
                         "peak_kind": f"{kind} (HBM copy bandwidth)", "bytes_per_lu": BYTES_PER_LU[STORAGE],
                         "kernel": kname,
                         "limiter": "FP32 operand bandwidth of the packed arithmetic (the FMA pipe) and the "
                                    "warps' rounds over 1216 places, not HBM"},
            "cpu_baseline": cpu,
            "e2e": {"value": round(e2e_val, 2), "unit": UNIT, "h2d_bytes_per_step": int(h2d),
                    "d2h_bytes_per_step": int(d2h),
                    "path": "amlbm_batch_init_all_f32 (pinned FP32 host arrays, all 64 instances) + "
                            "amlbm_batch_step(1) + amlbm_batch_diagnostics_all"},
            "e2e_fp64_inputs": {"value": round(e2e64_val, 2), "unit": UNIT, "h2d_bytes_per_step": int(h2d64),
                                "d2h_bytes_per_step": int(d2h),
                                "path": "amlbm_batch_init_all (pinned FP64 host arrays) + amlbm_batch_step(1) + "
                                        "amlbm_batch_diagnostics_all"},
            "gpu_launches": args.steps * lps,
            "clocks": clk.summary(),
            "graph_back_to_back": graph,
            "compare_mlups": compare or None,
            "adjoint": adjoint if (rank == 0 and not args.no_compare) else None,
            "scaled_hbm_cases": scaled if (rank == 0 and not args.no_compare) else None,
            "precision_vs_f64": precision if (rank == 0 and not args.no_compare) else None,
            "wall_s_timed_loop": round(wall, 3),
            "five_chunks_of_timed_steps": five,
        }
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()


CTYPE = {"f64": "double", "f32": "float", "f16": "__half", "bf16": "__nv_bfloat16"}


def kernel_name(storage, sched, tile):
    """The step kernel a batch of this storage, schedule and tile launches, and the
    source file that holds it."""
    t = CTYPE[storage]
    csrc = os.path.join(ROOT, "paper_1310_1871_gb300", "csrc")
    if sched == "pair" and tile[0] == 48 and storage != "f64":  # strips of tile[1] rows
        return f"strip_step<{t}>, {tile[1]} rows", os.path.join(csrc, "amlbm_step_strip.cu")
    if sched == "pair":
        return f"pair_persistent<{t}, {tile[0]}, {tile[1]}>", os.path.join(csrc, "amlbm_step_pair.cu")
    if sched == "fused" and tile[0] == 26 and tile[1] <= 10 and storage != "f64":
        return f"row_kernel<{t}>, {tile[1]} rows", os.path.join(csrc, "amlbm_step_row.cu")
    if sched == "split" and storage == "f64":
        return f"f64_stream<{tile[0]}, {tile[1]}> + f64_force", os.path.join(csrc, "amlbm_step_split64.cu")
    if sched == "fused":
        return f"lbm_persistent<{t}, {tile[0]}, {tile[1]}>", os.path.join(csrc, "amlbm_step.cu")
    return f"stream_kernel<{t}, {tile[0]}, {tile[1]}> + force_kernel", os.path.join(csrc, "amlbm_step.cu")


def graph_back_to_back(torch, rank, stream, steps, tile="auto", schedule="auto", chunk=20):
    """The headline form's steps replayed back to back from captured CUDA graphs of
    `chunk` timesteps each (amlbm_batch_step with graph_chunk): no L2 flush between
    steps, so the state stays L2-resident; CUDA events around all `steps`."""
    steps = max(chunk, steps // chunk * chunk)
    b, _ = build_batch(STORAGE, rank, tile=tile, graph_chunk=chunk, stream=stream, schedule=schedule)
    b.step(3 * chunk)  # warm-up (captures the graphs of both parities)
    torch.cuda.synchronize()
    a, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record(stream)
    b.step(steps)
    e.record(stream)
    torch.cuda.synchronize()
    ms = a.elapsed_time(e) / steps
    out = {"mlups": round(b.sites / (ms * 1e-3) / 1e6, 1), "ms_per_step": round(ms, 6), "steps": steps,
           "graph_chunk": chunk, "l2": "not flushed (state L2-resident)",
           "launch": "amlbm_batch_step replaying captured CUDA graphs of 20 timesteps",
           "schedule": b.schedule, "tile": list(b.tile)}
    b.close()
    return out


def adjoint_cost(torch, T=10000):
    """Cost of the discrete adjoint on the differentiable drop (512 x 128, R = 48, 16
    Legendre amplitudes, a2^2 objective, checkpoints every 100 steps), FP32 and FP64:
    wall time of amlbm_adjoint (forward with checkpoints + recomputation + reverse
    sweep) over the wall time of the forward run alone."""
    from paper_1310_1871_gb300 import amlbm
    amps = I.legendre_amplitudes(16, 0.02, seed=2024)
    out = {"workload": "differentiable drop 512 x 128, R=48, 16 amplitudes, J = a2(T)^2", "T": T,
           "ckpt_every": 100}
    for st in ("f32", "f64"):
        lat = amlbm.Lattice(512, 128, tau=1.0, G=-5.0, storage=st)
        lat.objective(200, amps, 256.0, 48.0)  # warm-up (kernel attributes, workspace)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        lat.objective(T, amps, 256.0, 48.0)
        torch.cuda.synchronize()
        tf = time.perf_counter() - t0
        t0 = time.perf_counter()
        lat.adjoint(T, amps, 256.0, 48.0, ckpt_every=100)
        torch.cuda.synchronize()
        ta = time.perf_counter() - t0
        out[st] = {"forward_s": round(tf, 4), "adjoint_s": round(ta, 4), "ratio": round(ta / tf, 2)}
        lat.close()
    return out


def precision_vs_f64(torch, steps=1000):
    """Per-instance max relative rho error of the reduced-precision forms against
    the FP64 form after `steps` timesteps of the 64-drop sweep, and their
    throughput on the same sweep (back-to-back steps, autotuned launch).
    Instances whose FP64 run itself goes non-finite (the unstable corner of the
    parameter ranges) are left out and counted."""
    from paper_1310_1871_gb300 import amlbm
    inst = I.batch_sweep(64)
    cols = [np.concatenate([np.ravel(x.make_fields()[q]) for x in inst]) for q in range(3)]

    def run(storage, shift, rounding="default"):
        specs = [amlbm.InstanceSpec(x.Nz, x.Nr, x.tau, x.G, shift=shift, rounding=rounding) for x in inst]
        b = amlbm.Batch(specs, storage=storage, tile="auto")
        b.init_all(*cols)
        torch.cuda.synchronize()
        a, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        b.step(steps)
        e.record()
        torch.cuda.synchronize()
        ms = a.elapsed_time(e) / steps
        rho = [b.read(k)[0] for k in range(len(inst))]
        b.close()
        return rho, b.sites / (ms * 1e-3) / 1e6
    ref, ref_mlups = run("f64", "default")
    ok = [k for k in range(len(inst)) if np.isfinite(ref[k]).all()]
    out = {"steps": steps, "instances_compared": len(ok), "unstable_in_f64": len(inst) - len(ok),
           "f64_mlups": round(ref_mlups, 1)}
    for storage, shift, rounding in (("f32", "default", "default"), ("bf16", "default", "default"),
                                     ("bf16", "equilibrium", "default"), ("f16", "default", "default"),
                                     ("f16", "equilibrium", "default"), ("f16", "equilibrium", "stochastic")):
        rho, mlups = run(storage, shift, rounding)
        err = [float(np.abs(rho[k] / ref[k] - 1).max()) for k in ok]
        key = f"{storage}/{shift}" + ("/stochastic" if rounding == "stochastic" else "")
        out[key] = {"max_rel_rho_err": float(f"{max(err):.3e}"), "meets_1e-4": max(err) <= 1e-4,
                                     "median_rel_rho_err": float(f"{float(np.median(err)):.3e}"),
                                     "mlups": round(mlups, 1), "over_f64": round(mlups / ref_mlups, 2)}
    return out


def scaled_cases(torch, tile, sched, steps=10):
    """The HBM-sized cases: the oscillating-drop physics (G = -5, tau = 1, P2
    perturbation 5 %) scaled 32x to an 8192 x 4096 lattice (33.5 M sites, R = 1280),
    and the sweep's recipe with 1024 instances (seeds 1234 + k).  The headline storage form.
    Each state is far larger than L2, so back-to-back steps read it from HBM;
    CUDA events around `steps` timesteps after 3 warm-up steps."""
    from paper_1310_1871_gb300 import amlbm
    hbm, kind = peaks()
    out = {}

    def timed(step_fn, sites):
        for _ in range(3):
            step_fn()
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(steps):
            step_fn()
        b.record()
        torch.cuda.synchronize()
        ms = a.elapsed_time(b) / steps
        gbs = BYTES_PER_LU[STORAGE] * sites / (ms * 1e-3) / 1e9
        return {"sites": int(sites), "ms_per_step": round(ms, 4), "mlups": round(sites / (ms * 1e-3) / 1e6, 1),
                "achieved_gbs": round(gbs, 1), "frac_of_measured_hbm": round(gbs / hbm, 4)}

    Nz, Nr, R = 8192, 4096, 1280.0
    lat = amlbm.Lattice(Nz, Nr, tau=1.0, G=-5.0, storage=STORAGE)
    z = torch.arange(Nz, dtype=torch.float64, device="cuda")[None, :] - Nz / 2
    r = torch.arange(Nr, dtype=torch.float64, device="cuda")[:, None] + 0.5
    d = torch.sqrt(z * z + r * r)
    ct = z / d
    rs = R * (1.0 + 0.05 * 0.5 * (3 * ct * ct - 1))
    rho = I.RHO_V_G5 + 0.5 * (I.RHO_L_G5 - I.RHO_V_G5) * (1 - torch.tanh((d - rs) / 2.0))
    lat.init_fields_device(rho.contiguous())
    del z, r, d, ct, rs, rho
    out["lattice_8192x4096"] = timed(lambda: lat.step(1), Nz * Nr)
    lat.close()

    inst = I.batch_sweep(1024)
    specs = [amlbm.InstanceSpec(x.Nz, x.Nr, x.tau, x.G) for x in inst]
    b = amlbm.Batch(specs, storage=STORAGE, tile=tuple(tile), schedule=sched)
    cols = [np.concatenate([np.ravel(x.make_fields()[q]) for x in inst]) for q in range(3)]
    b.init_all(*cols)
    out["batch_1024"] = dict(timed(lambda: b.step(1), b.sites), tile=list(b.tile), schedule=b.schedule)
    b.close()
    out["peak"] = f"{hbm} GB/s ({kind} HBM copy bandwidth)"
    return out


def cpu_model():
    """The host CPU's model name (lscpu, else /proc/cpuinfo), for the baseline record."""
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for ln in out.splitlines():
            if ln.strip().startswith("Model name:"):
                return ln.split(":", 1)[1].strip()
    except (OSError, subprocess.SubprocessError):
        pass
    try:
        for ln in open("/proc/cpuinfo"):
            if ln.lower().startswith(("model name", "cpu part")):
                return ln.split(":", 1)[1].strip()
    except OSError:
        pass
    import platform
    return platform.processor() or platform.machine()


def host_cores():
    """Cores this process may run on."""
    try:
        return len(os.sched_getaffinity(0))
    except AttributeError:
        return os.cpu_count() or 1


def oracle_mlups(seconds, omp):
    """The FP64 oracle stepping the sweep's instances in turn (one instance-timestep per
    step) until about `seconds` of work is done: (MLUPS, steps, site updates, seconds,
    threads).  omp: the OpenMP build (its site loops over all host cores)."""
    import oracle as O
    nthreads = O.threads(host_cores()) if omp else 1
    inst = I.batch_sweep(64)
    states = {}
    done_sites = 0
    elapsed = 0.0
    k = 0
    while elapsed < seconds:
        x = inst[k % 64]
        if k % 64 not in states:
            o = O.Oracle(x.Nz, x.Nr, tau=x.tau, G=x.G, omp=omp)
            states[k % 64] = (o, o.init(*x.make_fields()))
        o, f = states[k % 64]
        t1 = time.perf_counter()
        f = o.run(f, 1)
        elapsed += time.perf_counter() - t1
        states[k % 64] = (o, f)
        done_sites += x.Nz * x.Nr
        k += 1
    return done_sites / elapsed / 1e6, k, done_sites, elapsed, nthreads


def cpu_baseline(seconds=15.0):
    """The FP64 oracle on the host, on one thread and with its OpenMP build on every
    core, each for about `seconds` of the sweep's instance-timesteps."""
    v1, n1, s1, e1, _ = oracle_mlups(seconds, omp=False)
    vn, nn, sn, en, thr = oracle_mlups(seconds, omp=True)
    model = cpu_model()
    return {"value": round(vn, 3), "unit": UNIT, "cores": thr, "kind": "oracle",
            "sample": f"{nn} instance-timesteps of the 64-drop sweep in turn ({sn} site updates, "
                      f"{en:.1f} s), FP64, OpenMP over lattice rows on {thr} threads",
            "single_thread": {"value": round(v1, 3), "cores": 1,
                              "sample": f"{n1} instance-timesteps ({s1} site updates, {e1:.1f} s)"},
            "cpu_model": model}


def run_reference(args):
    """The oracle as the reference arm, on every host core (its OpenMP build): each
    step advances one instance of the sweep (in turn) by one timestep; MLUPS over the
    timed steps."""
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    import oracle as O
    thr = O.threads(host_cores())
    inst = I.batch_sweep(64)
    states = []
    for x in inst:
        o = O.Oracle(x.Nz, x.Nr, tau=x.tau, G=x.G, omp=True)
        states.append([o, o.init(*x.make_fields())])
    for s in range(args.warmup):
        o, f = states[s % 64]
        states[s % 64][1] = o.run(f, 1)
    sites = 0
    t0 = time.perf_counter()
    for s in range(args.steps):
        o, f = states[(args.warmup + s) % 64]
        states[(args.warmup + s) % 64][1] = o.run(f, 1)
        sites += inst[(args.warmup + s) % 64].Nz * inst[(args.warmup + s) % 64].Nr
    el = time.perf_counter() - t0
    val = sites / el / 1e6
    line = {
        "metric": METRIC, "value": round(val, 3), "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": round(el / max(args.steps, 1) * 1e3, 4),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic", "impl": "reference",
        "config": dict(config(sum(x.Nz * x.Nr for x in inst), "f64"),
                       l2="host caches (the oracle runs on the host cores)",
                       launch="FP64 oracle, one instance-timestep of the sweep per step, instances in turn"),
        "cpu_baseline": {"value": round(val, 3), "unit": UNIT, "cores": thr, "kind": "oracle",
                         "sample": f"one instance-timestep of the 64-drop sweep per step, instances in "
                                   f"turn ({sites} site updates in {el:.1f} s), FP64 oracle, OpenMP "
                                   f"over lattice rows on {thr} threads", "cpu_model": cpu_model()},
        "e2e": {"value": round(val, 3), "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3000)
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--impl", default="amlbm", choices=["amlbm", "reference"])
    ap.add_argument("--no-cpu", action="store_true", help="skip the oracle CPU baseline")
    ap.add_argument("--no-compare", action="store_true", help="skip the FP64/FP32 comparison runs")
    ap.add_argument("--cpu-seconds", type=float, default=10.0)
    ap.add_argument("--launch", default="auto",
                    help="launch of the timed batch: auto (the autotuner's choice) or SCHEDULE:TZxTR, "
                         "e.g. pair:32x16")
    args = ap.parse_args()
    if args.warmup < 3:
        ap.error("--warmup must be at least 3")
    if args.impl == "reference":
        run_reference(args)
    else:
        run_gpu(args)


if __name__ == "__main__":
    main()
