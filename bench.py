#!/usr/bin/env python
"""Benchmark of the GB300 MLS-MPM step + adjoint.

One bench step = one whole trajectory of the long-horizon dam-break scene
(2,000,000 particles: 1.4M water, 0.6M von Mises; 256^3 grid): set the initial
state, 1000 forward MPM steps (checkpoint every 50), the final-position loss,
and the full reverse sweep (recompute from checkpoints + hand-written adjoint
kernels) down to the gradients w.r.t. the initial positions. It is the
largest single-GPU workload of the build target; the 200k-particle
three-material tool scene (200 steps, grid-mass loss, gradients w.r.t. the
tool's actions), the 64 batched scenes, the surrogate, gradient sharing and
the gas solver are objects of the same line.

`value` = particle-steps per second of forward + adjoint with the inputs
resident in HBM; `e2e` = the same through the C-ABI with host buffers (copies
inside the timed region). One JSON line on rank 0.

  python bench.py [--gpus N --steps K --warmup W] [--impl reference]
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

METRIC = "particle-steps/s fwd and fwd+adjoint on 1 GB300, % HBM roofline, grad rel-err"
UNIT = "particle-steps/s (fwd+adjoint)"
WORKLOAD = ("dam break: 2,000,000 particles (1.4M water column, 0.6M von Mises blocks), 256^3 grid, "
            "1000 FP32 steps forward + adjoint of a final-position loss w.r.t. the initial positions, "
            "checkpoint every 50 (recompute from checkpoints)")
WORKLOAD_C2 = ("three-material tool scene: 200,000 particles (100k liquid, 60k von Mises, "
               "40k Drucker-Prager), 128^3 grid, kinematic box tool, 200 FP32 steps forward + "
               "adjoint of a grid-mass loss w.r.t. 20x6 actions, checkpoint every 20")


def max_over_ranks(values, world, device=None):
    """Each timed quantity (a list of floats) as its maximum over the ranks:
    the job is as slow as its slowest replica. Identity at world == 1; at
    world > 1 every rank gets the same maxima (all-reduce MAX in FP64 on the
    given device: the rank's GPU under NCCL, the CPU under gloo)."""
    if world <= 1:
        return [float(v) for v in values]
    import torch
    t = torch.tensor([float(v) for v in values], dtype=torch.float64, device=device)
    torch.distributed.all_reduce(t, op=torch.distributed.ReduceOp.MAX)
    return [float(v) for v in t.cpu()]


def whole_job_rate(units_per_rank, world, seconds_per_step):
    """Whole-job throughput: the units all replicas processed per step divided
    by the (max-over-ranks) time of a step."""
    return float(units_per_rank) * world / seconds_per_step


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--scale", type=float, default=1.0, help="particle-count scale (1.0 = the workload)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--launch", default=None,
                    help="scatter,gather,grid_blocks,resort,fuse[,persistent[,stage[,ctas]]] launch shapes instead of the autotuner "
                         "(e.g. for profilers: no tuning launches before the measured ones)")
    ap.add_argument("--profile-only", action="store_true",
                    help="run warm-up + K steps only (for external profilers)")
    ap.add_argument("--workload", default="line",
                    choices=["line", "multi_material", "dam_break", "surrogate", "surrogate_speed", "batched",
                             "gas", "rigid"],
                    help="line: the bench line (dam-break headline and every object). dam_break / "
                         "multi_material: that trajectory benchmark alone. surrogate: generate frames from "
                         "64-scene rollouts, train the conv surrogate, report its held-out error, error gate "
                         "and speed against the simulation. surrogate_speed: only the surrogate's kernel "
                         "speed (the `surrogate` object of the default line). batched: the 64-scene batched "
                         "launch (the `batched` object of the default line). rigid: the bench scene with "
                         "its sand block made a particle-represented rigid body")
    ap.add_argument("--grid-n", type=int, default=0,
                    help="dam_break / multi_material workload alone: grid nodes per axis (0 = the workload's)")
    ap.add_argument("--horizon", type=int, default=0,
                    help="dam_break / multi_material workload alone: steps per trajectory (0 = the workload's)")
    ap.add_argument("--checkpoint-every", type=int, default=0,
                    help="dam_break / multi_material workload alone: checkpoint interval (0 = the workload's)")
    ap.add_argument("--no-extras", action="store_true",
                    help="skip the objects of the default line after the headline")
    ap.add_argument("--no-surrogate-accuracy", action="store_true",
                    help="skip the surrogate's training and held-out accuracy object of the default line")
    ap.add_argument("--sur-rollouts", type=int, default=4, help="surrogate: 64-scene rollouts of frames")
    ap.add_argument("--sur-rollout-steps", type=int, default=88, help="surrogate: steps per rollout")
    ap.add_argument("--sur-train-steps", type=int, default=3000, help="surrogate: Adam steps")
    ap.add_argument("--sur-batch", type=int, default=8, help="surrogate: frames per Adam step")
    ap.add_argument("--sur-lr", type=float, default=1e-3)
    ap.add_argument("--sur-save", default=None, help="surrogate: write the trained parameters (float32) here")
    ap.add_argument("--sur-bound", type=float, default=0.1,
                    help="surrogate: relative L2 error above which the gate falls back to the simulation")
    return ap.parse_args()


def profiled_traffic(kernel, workload=None):
    """DRAM bytes per full-size launch of `kernel` on `workload` recorded in a
    profiles/ summary, if it was captured from the current CUDA sources (else
    None)."""
    return profiled_value(kernel, "traffic_per_launch_full_size", workload)


def profiled_value(kernel, key, workload=None):
    """A per-launch figure (`key`: traffic_per_launch_full_size,
    instructions_per_launch_full_size) of `kernel` recorded in a profiles/
    summary, if it was captured from the current CUDA sources (else None).
    A record line may name its workload (`workload=...`); with `workload`
    given, only a record of that workload (or one naming none) counts."""
    import re
    from paper_2303_02346_gb300 import build as b
    if kernel.startswith("sur_"):
        group = "surrogate"
    elif kernel.startswith("gas_"):
        group = "gas"
    elif kernel in ("g2p_adj", "grid_adj", "p2g_adj", "adj_fused"):
        group = "mpm_adj"
    else:
        group = "mpm_fwd"
    cur = b.source_hash(group)
    pdir = os.path.join(ROOT, "profiles")
    if not os.path.isdir(pdir):
        return None
    for name in sorted(os.listdir(pdir)):
        with open(os.path.join(pdir, name)) as f:
            for line in f:
                m = re.match(key + r":\s*(\d+)\s+kernel=(\S+)\s+source_hash=(\S+)(?:\s+workload=(\S+))?",
                             line)
                if m and m.group(2) == kernel and m.group(3) == cur and (
                        workload is None or m.group(4) in (None, workload)):
                    return int(m.group(1))
    return None


def issue_roofline(kernel, ms_avg, workload=None):
    """The kernel's instruction issue rate against the GB300's: warp
    instructions per launch (ncu, scaled to the full-size launch) over the mean
    launch time, against 152 SMs x 4 schedulers x one warp instruction per
    cycle at the maximum SM clock. None without a current profile."""
    inst = profiled_value(kernel, "instructions_per_launch_full_size", workload)
    if inst is None:
        return None
    mhz = 2070.0
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            mhz = float(json.load(f).get("sm_max_mhz", mhz))
    achieved = inst / (ms_avg / 1e3)
    peak = 152 * 4 * mhz * 1e6
    return {"warp_instructions_per_launch": inst, "achieved": round(achieved / 1e9, 1),
            "peak": round(peak / 1e9, 1), "unit": "G warp-instructions/s", "frac": round(achieved / peak, 4)}


def load_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


def load_tensor_peak(sustained=False):
    """Dense BF16 tensor peak in TFLOP/s (burst for a kernel timed in short
    runs, sustained for long loops)."""
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        key = "bf16_tflops_sustained" if sustained else "bf16_tflops"
        if key in d:
            return float(d[key]), "measured"
    return (1700.0 if sustained else 1900.0), "fallback"


# ----------------------------------------------------------------------------
# clocks
# ----------------------------------------------------------------------------
CLOCK_Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
           "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
           "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")


def _clock_rows(path):
    rows = []
    with open(path) as f:
        for line in f:
            parts = [p.strip() for p in line.split(",")]
            if len(parts) >= 9:
                rows.append(parts)
    return rows


def start_clocks(gpu_index):
    """Start an nvidia-smi sampler (every 100 ms) and wait until it has
    written its first row, so that the timed region that follows is covered;
    returns (process, csv path, rows to skip = those taken before the timed
    region)."""
    fd, path = tempfile.mkstemp(suffix=".csv")
    os.close(fd)
    try:
        proc = subprocess.Popen(["nvidia-smi", f"--id={gpu_index}", f"--query-gpu={CLOCK_Q}",
                                 "--format=csv,noheader,nounits", "-lms", "100"],
                                stdout=open(path, "w"), stderr=subprocess.DEVNULL)
    except Exception:
        return None, path, 0
    t0 = time.time()
    while time.time() - t0 < 5.0 and proc.poll() is None and not _clock_rows(path):
        time.sleep(0.02)
    return proc, path, len(_clock_rows(path))


def stop_clocks(proc, path, skip=0):
    if proc is None:
        return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
    proc.terminate()
    try:
        proc.wait(timeout=5)
    except Exception:
        proc.kill()
    rows = _clock_rows(path)
    os.unlink(path)
    # samples taken inside the timed region; the last one before it when the
    # region was shorter than one sampling interval
    rows = rows[skip:] or rows[-1:]
    if not rows:
        return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}

    def num(x):
        try:
            return float(x)
        except ValueError:
            return None

    sm = [num(r[1]) for r in rows if num(r[1]) is not None]
    mx = max((num(r[2]) or 0.0) for r in rows)
    under = [s for s in sm if s > 0.5 * mx] or sm
    names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
    reasons = sorted({names[i] for r in rows for i in range(4) if r[5 + i].lower().startswith("active")})
    return {"sm_mhz": statistics.median(under) if under else None, "sm_max_mhz": mx,
            "reasons": reasons, "samples": len(rows)}


# ----------------------------------------------------------------------------
# algorithmic bytes per kernel launch: per-particle state bytes by material
# (liquid, solid) and bytes per active grid node (16 B per float4 node record)
# ----------------------------------------------------------------------------
def algorithmic_bytes(kernel, n_liq, n_sol, nodes):
    per = {
        # read x v C + F (solid) / J (liquid) + tag, write F_p (solid) | grid write
        "p2g": (64 + 4, 96 + 4 + 36, 16),
        # read x + tag + F_p / J, gather grid, write x v C F / J
        "g2p": (16 + 4 + 60 + 4, 16 + 36 + 60 + 36, 16),
        # G2P of step n-1 + P2G of step n: read x tag F_p/J, write x v C F/J and
        # F_p (solid) | grid gather + grid write
        "g2p2g": (12 + 4 + 4 + 60 + 4, 12 + 4 + 36 + 60 + 36 + 36, 32),
        # read acc, write gv, zero acc
        "grid_update": (0, 0, 48),
        # one step of the persistent forward (per step): the lean fused step
        # (read x tag F_p/J, write x J / x F_p) and the grid update | grid
        # gather, grid write, grid update
        "fwd_run": (12 + 4 + 4 + 12 + 4, 12 + 4 + 36 + 12 + 36, 32 + 48),
        # read x tag C' F, read adj (x v C F), gather gv, write xbar, scatter vbar
        "g2p_adj": (12 + 4 + 36 + 4 + 64 + 12, 12 + 4 + 36 + 36 + 96 + 12, 32),
        # read vbar, zero it, read (u, m), write (mbar, mvbar)
        "grid_adj": (0, 0, 64),
        # read x v C F tag C', read xbar Fbar, gather gadj, write adj
        "p2g_adj": (64 + 4 + 36 + 12 + 4 + 64, 96 + 4 + 36 + 12 + 36 + 96, 16),
        # P2G adjoint of step n + G2P adjoint of step n-1: read state n (x v C, F),
        # C^{n+1}, x^{n-1} (+J), F_p^{n-1}, xbar Fbar; write xbar Fbar | gather
        # gadj_m and gv, scatter vbar
        "adj_fused": (60 + 4 + 4 + 36 + 16 + 12 + 4 + 12 + 4, 60 + 4 + 84 + 36 + 12 + 36 + 12 + 36 + 12 + 36, 48),
    }
    if kernel not in per:
        return None
    a, b, c = per[kernel]
    return n_liq * a + n_sol * b + nodes * c


# ----------------------------------------------------------------------------
# algorithmic bytes of one particle-step: the state round trip (x, v, C and
# J or F read and written: 2 x 64 B for a liquid, 2 x 96 B for a solid) plus
# about 6 B of grid per particle; the adjoint of a step reads the state and
# the next step's adjoint and writes this step's adjoint (3 x 64 / 3 x 96 B)
# plus about three times the grid bytes
# ----------------------------------------------------------------------------
STEP_BYTES = {"g2p2g": (134, 198), "fwd_run": (134, 198), "adj_fused": (210, 306)}
STEP_BYTES_WHAT = {
    "g2p2g": "one particle-step of state read + write (x v C J: 2 x 64 B liquid; x v C F: 2 x 96 B solid) "
             "+ 6 B of grid per particle",
    "adj_fused": "one particle-step of adjoint (state read, next adjoint read, adjoint write: 3 x 64 B liquid, "
                 "3 x 96 B solid) + 18 B of grid per particle",
}
STEP_BYTES_WHAT["fwd_run"] = STEP_BYTES_WHAT["g2p2g"] + " (per step of the persistent run)"

FWD_KERNELS = ("p2g", "g2p2g", "g2p", "grid_update", "sort", "rigid", "fwd_run")
ADJ_KERNELS = ("g2p_adj", "p2g_adj", "adj_fused", "grid_adj", "permute", "tool_adj", "seed", "rigid_adj")


def _merge(dst, prof):
    for k, (ms, n) in prof.items():
        a = dst.setdefault(k, [0.0, 0])
        a[0] += ms
        a[1] += n


def run_trajectory(args, sc, dev, rank, world, steps, warmup, e2e=True, clocks=True, label=None):
    """One bench step = one whole trajectory of scene `sc`: set the initial
    state (and the tool), sc.n_steps MPM steps forward with a checkpoint every
    sc.checkpoint_every steps, the scene's loss on the final state, and the
    reverse sweep (recompute from checkpoints + hand-written adjoints) down to
    the gradients w.r.t. the initial state (and the tool's actions). Returns
    the timings (CUDA events on the library's stream, max over ranks), the
    per-kernel event timings of a serial pass, the roofline of the dominant
    step kernel, device memory and the recompute overhead."""
    import torch

    from paper_2303_02346_gb300 import binding as B
    from paper_2303_02346_gb300.simulator import Simulator
    T, N = sc.n_steps, sc.n_particles
    liquid = [i for i, m in enumerate(sc.materials) if m.kind in (0, 4)]
    n_liq = int(sum(int((sc.mat == i).sum()) for i in liquid))
    n_sol = N - n_liq
    torch.cuda.synchronize()
    free0, total = torch.cuda.mem_get_info(dev)
    sim = Simulator(sc, device=dev)
    h = sim.h
    x0 = torch.tensor(sc.x, dtype=torch.float32, device=dev)
    v0 = torch.tensor(sc.v, dtype=torch.float32, device=dev)
    mat = torch.tensor(sc.mat, dtype=torch.uint8, device=dev)
    tool = bool(sc.tool_enabled)
    if tool:
        pose0 = torch.tensor(sc.tool_pose0, dtype=torch.float32, device=dev)
        acts = torch.tensor(sc.tool_actions, dtype=torch.float32, device=dev)
        ga = torch.empty(sc.n_scenes, acts.shape[1], 6, dtype=torch.float32, device=dev)
    L = sc.loss
    if L["kind"] == "position":
        def loss():
            B.sim_position_loss(h, -1, L["target"], L.get("weight", 1.0), n_out=sc.n_scenes)
        loss_what = "final-position loss"
    else:
        tm = torch.tensor(L["target_mass"], dtype=torch.float32, device=dev)
        td = torch.tensor(L["target_dist"], dtype=torch.float32, device=dev)
        M = float(L["total_mass"])

        def loss():
            B.sim_grid_mass_loss(h, 0, tm, td, M)
        loss_what = "grid-mass loss"
    gx = torch.empty(N, 3, dtype=torch.float32, device=dev)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    stream = torch.cuda.current_stream(dev)

    def start():
        B.sim_set_particles(h, -1, x0, v0, mat)
        if tool:
            B.sim_set_tool(h, -1, pose0, acts, acts.shape[1])

    def trajectory(ev_f=None):
        start()
        if ev_f is not None:
            ev_f[0].record(stream)
        B.sim_step(h, T)
        if ev_f is not None:
            ev_f[1].record(stream)
        loss()
        B.sim_backward(h, gx, None, ga if tool else None)

    # launch shapes picked by the library's autotuner on this scene (untimed)
    start()
    if args.launch:
        tuning = tuple(int(v) for v in args.launch.split(","))
        B.sim_set_launch(h, *tuning)
    else:
        tuning = B.sim_autotune(h, 20)
    for _ in range(warmup):
        trajectory()
    torch.cuda.synchronize()
    free1, _ = torch.cuda.mem_get_info(dev)
    if world > 1:
        torch.distributed.barrier()
    if args.profile_only:
        for _ in range(steps):
            trajectory()
        torch.cuda.synchronize()
        sim.close()
        return None

    clk, clk_path, clk_skip = start_clocks(dev.index) if (clocks and rank == 0) else (None, None, 0)
    launches0 = B.sim_kernel_launches(h)
    times, ftimes = [], []
    torch.cuda.synchronize()
    if world > 1:
        torch.distributed.barrier()
    for _ in range(steps):
        flush.zero_()  # untimed L2 flush between timed steps
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        f0, f1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        trajectory((f0, f1))
        e1.record(stream)
        torch.cuda.synchronize()
        times.append(e0.elapsed_time(e1))
        ftimes.append(f0.elapsed_time(f1))
    torch.cuda.synchronize()
    if world > 1:
        torch.distributed.barrier()
    launches = B.sim_kernel_launches(h) - launches0
    clk_out = stop_clocks(clk, clk_path, clk_skip) if (clocks and rank == 0) else None
    total_ms, fwd_ms = max_over_ranks([sum(times), sum(ftimes)], world, dev)
    ms_per_step = total_ms / steps
    value = whole_job_rate(float(N) * T, world, ms_per_step / 1e3)
    fwd_value = whole_job_rate(float(N) * T, world, fwd_ms / steps / 1e3)

    # per-kernel event timings of serial passes (no graphs, no overlapped
    # recompute): the forward (sim_step) and the backward (recompute + adjoint)
    # recorded apart
    reps = max(1, min(steps, 3))
    fwd_prof, bwd_prof = {}, {}
    for _ in range(reps):
        flush.zero_()
        B.sim_profile_enable(h, 1)
        start()
        B.sim_step(h, T)
        _merge(fwd_prof, B.sim_profile_read(h))
        B.sim_profile_enable(h, 1)
        loss()
        B.sim_backward(h, gx, None, ga if tool else None)
        _merge(bwd_prof, B.sim_profile_read(h))
    B.sim_profile_enable(h, 0)
    kern = {}
    _merge(kern, fwd_prof)
    _merge(kern, bwd_prof)
    kern = {k: {"ms_total": round(v[0] / reps, 4), "launches": v[1] // reps, "ms_avg": round(v[0] / max(v[1], 1), 5)}
            for k, v in kern.items()}
    fwd_k = sum(v[0] for k, v in fwd_prof.items() if k in FWD_KERNELS) / reps
    rec_k = sum(v[0] for k, v in bwd_prof.items() if k in FWD_KERNELS) / reps
    adj_k = sum(v[0] for k, v in bwd_prof.items() if k in ADJ_KERNELS) / reps
    peak, peak_kind = load_peaks()
    dom = max((k for k in kern if k in STEP_BYTES), key=lambda k: kern[k]["ms_total"])
    per_liq, per_sol = STEP_BYTES[dom]
    abytes = n_liq * per_liq + n_sol * per_sol
    achieved = abytes / (kern[dom]["ms_avg"] / 1e3) / 1e9
    tag = label or sc.name
    roofline = {"bound": "hbm", "kernel": dom, "achieved": round(achieved, 1), "peak": peak,
                "peak_source": peak_kind, "unit": "GB/s", "frac": round(achieved / peak, 4),
                "traffic": profiled_traffic(dom, tag), "algorithmic_bytes_per_launch": abytes,
                "bytes_basis": STEP_BYTES_WHAT[dom], "avg_launch_ms": kern[dom]["ms_avg"],
                "kernel_bytes_per_launch": algorithmic_bytes(dom, n_liq, n_sol, estimate_active_nodes(sc))}
    issue = issue_roofline(dom, kern[dom]["ms_avg"], tag)
    if issue is not None:
        roofline["issue"] = issue
    # state sizes per particle-step for forward + adjoint under checkpointing:
    # forward 2, adjoint 3, and 2 for each step the backward recomputes (a
    # recomputed step is a P2G or a fused G2P -> P2G of the serial pass)
    rec_steps = min(T, (bwd_prof.get("g2p2g", (0.0, 0))[1] + bwd_prof.get("p2g", (0.0, 0))[1]) // reps)
    sizes = 5 + 2 * rec_steps / T
    step_bytes = int(round(sizes * (64 * n_liq + 96 * n_sol) * T))
    out = {
        "value": round(value, 1), "ms_per_step": round(ms_per_step, 3),
        "fwd": {"value": round(fwd_value, 1), "unit": "particle-steps/s (forward only)",
                "ms_per_trajectory": round(fwd_ms / steps, 3)},
        "bwd_ms_per_trajectory": round((total_ms - fwd_ms) / steps, 3),
        "roofline": roofline,
        "trajectory_roofline": {"bytes": step_bytes,
                                "basis": f"{sizes:.3f} state sizes per particle-step (forward 2, adjoint 3, "
                                         f"recompute 2 x {rec_steps} of {T} steps; 64 B liquid, 96 B solid)",
                                "achieved": round(step_bytes / (ms_per_step / 1e3) / 1e9, 1), "unit": "GB/s",
                                "frac": round(step_bytes / (ms_per_step / 1e3) / 1e9 / peak, 4)},
        "kernels": kern,
        "gpu_launches": int(launches),
        "memory": {"handle_device_bytes": int(free0 - free1), "device_bytes_total": int(total),
                   "peak_device_bytes_in_use": int(total - free1)},
        "recompute": {"forward_kernel_ms": round(fwd_k, 3), "recompute_kernel_ms": round(rec_k, 3),
                      "adjoint_kernel_ms": round(adj_k, 3),
                      "overhead": round(rec_k / max(fwd_k + adj_k, 1e-9), 4),
                      "what": "kernel time of the backward's forward recompute over the forward's and the "
                              "adjoint's kernel time (serial event-timed pass)"},
        "config": {"workload": sc.name, "particles": N, "liquid": n_liq, "solid": n_sol, "grid": sc.grid_n,
                   "scenes": sc.n_scenes, "trajectory_steps": T, "checkpoint_every": sc.checkpoint_every,
                   "loss": loss_what,
                   "l2": "256 MB buffer written (untimed) between timed steps; the per-trajectory working set "
                         "(checkpoints, chunk states, per-step grids) exceeds L2",
                   "launch": {"scatter_threads": tuning[0], "gather_threads": tuning[1],
                              "grid_blocks_per_cta": tuning[2], "fused_adjoint": bool(tuning[4]),
                              "persistent_forward": bool(tuning[5]) if len(tuning) > 5 else False,
                              "staged_gather": bool(tuning[6]) if len(tuning) > 6 else False,
                              "scatter_ctas_per_sm": tuning[7] if len(tuning) > 7 else 3,
                              "cuda_graphs": True, "autotuned": not args.launch}},
    }
    if clk_out is not None:
        out["clocks"] = clk_out
    if e2e and not args.no_e2e:
        out["e2e"] = run_e2e(args, sc, h, B, dev, T, N, world, steps)
    sim.close()
    return out


def run_ours(args, rank, world, local_rank):
    """The bench line: the 2M-particle long-horizon scene (the largest
    single-GPU workload) as the headline, then the 200k-particle three-material
    tool scene, the batched scenes, the surrogate, gradient sharing and the gas
    solver as objects of the same line (rank 0)."""
    import torch

    import scenes
    from paper_2303_02346_gb300 import build as b

    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    if rank == 0 or world == 1:
        b.build()
    if world > 1:
        torch.distributed.barrier()
    sc = scenes.dam_break(scale=args.scale)
    head = run_trajectory(args, sc, dev, rank, world, args.steps, args.warmup, label="dam_break")
    if head is None:
        return None
    out = {
        "metric": METRIC, "value": head["value"], "unit": UNIT, "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": head["ms_per_step"],
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
        "data": "synthetic (seeded scene generator; stands in for the paper's tasks at the largest stated size)",
        "config": dict(head["config"], workload=WORKLOAD,
                       parallelism="replicas" if world > 1 else "single"),
    }
    for k in ("fwd", "bwd_ms_per_trajectory", "roofline", "trajectory_roofline", "kernels", "gpu_launches",
              "memory", "recompute", "clocks", "e2e"):
        if k in head:
            out[k] = head[k]
    extras = rank == 0 and not args.no_extras
    if extras:
        mm = run_trajectory(args, scenes.multi_material(scale=args.scale), dev, rank, 1, max(args.steps, 5),
                            args.warmup, e2e=False, clocks=False, label="multi_material")
        mm["workload"] = WORKLOAD_C2
        out["multi_material"] = mm
        batched = run_batched(args, dev, steps=2, warmup=1)
        batched["vs_single_scene"] = round(batched["value"] / mm["value"], 3)
        out["batched"] = batched
        out["surrogate"] = run_surrogate_quick(args, dev)
        out["gpu_launches_surrogate_per_inference"] = out["surrogate"]["kernel_launches_per_inference"]
        out["sharing"] = run_sharing(args, dev)
        out["gas"] = run_gas(args, dev)
        if not args.no_surrogate_accuracy:
            out["surrogate_accuracy"] = run_surrogate(args, build=False)
    return out


# ----------------------------------------------------------------------------
# our implementation
# ----------------------------------------------------------------------------
def estimate_active_nodes(sc):
    """Nodes of the 4^3 grid blocks that the particles' stencils touch at the
    initial state (a lower bound of the per-step active set)."""
    import numpy as np
    n = sc.grid_n
    base = np.clip(np.floor(sc.x * n - 0.5).astype(int), 0, n - 3)
    blocks = set()
    for off in [(0, 0, 0), (2, 0, 0), (0, 2, 0), (0, 0, 2), (2, 2, 0), (2, 0, 2), (0, 2, 2), (2, 2, 2)]:
        bb = (base + np.array(off)) // 4
        blocks.update(map(tuple, np.unique(bb, axis=0)))
    return 64 * len(blocks)


def run_e2e(args, sc, h, B, dev, T, N, world, steps):
    """Same trajectory through the C-ABI with host buffers: pinned host inputs
    (initial state, tool, loss targets) copied in, and the loss and the
    gradient (w.r.t. the actions with a tool, else w.r.t. the initial
    positions) copied out, inside the timed region."""
    import torch
    pin = lambda a, dt: torch.tensor(a, dtype=dt).pin_memory()
    x0 = pin(sc.x, torch.float32)
    v0 = pin(sc.v, torch.float32)
    mat = pin(sc.mat, torch.uint8)
    ins = [x0, v0, mat]
    tool = bool(sc.tool_enabled)
    if tool:
        pose0 = pin(sc.tool_pose0, torch.float32)
        acts = pin(sc.tool_actions, torch.float32)
        grad = torch.empty(sc.n_scenes, acts.shape[1], 6, dtype=torch.float32).pin_memory()
        ins += [pose0, acts]
    else:
        grad = torch.empty(N, 3, dtype=torch.float32).pin_memory()
    L = sc.loss
    if L["kind"] == "position":
        tgt = np.asarray(L["target"], dtype=np.float32)
        ins_bytes = tgt.nbytes
        loss = lambda: B.sim_position_loss(h, -1, tgt, L.get("weight", 1.0), n_out=sc.n_scenes)
    else:
        tm = pin(L["target_mass"], torch.float32)
        td = pin(L["target_dist"], torch.float32)
        ins += [tm, td]
        ins_bytes = 0
        loss = lambda: B.sim_grid_mass_loss(h, 0, tm, td, float(L["total_mass"]))
    h2d = sum(t.numel() * t.element_size() for t in ins) + ins_bytes
    d2h = grad.numel() * grad.element_size() + 8 * (sc.n_scenes if L["kind"] == "position" else 1)

    def one():
        B.sim_set_particles(h, -1, x0, v0, mat)
        if tool:
            B.sim_set_tool(h, -1, pose0, acts, acts.shape[1])
        B.sim_step(h, T)
        loss()
        if tool:
            B.sim_backward(h, None, None, grad)
        else:
            B.sim_backward(h, grad, None, None)

    one()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(steps):
        one()
    torch.cuda.synchronize()
    dt = (time.perf_counter() - t0) / steps
    dt = max_over_ranks([dt], world, dev)[0]
    return {"value": round(whole_job_rate(N * T, world, dt), 1), "unit": UNIT, "h2d_bytes_per_step": int(h2d),
            "d2h_bytes_per_step": int(d2h), "ms_per_step": round(dt * 1e3, 3)}


# ----------------------------------------------------------------------------
# batched scenes in one launch
# ----------------------------------------------------------------------------
def run_batched(args, dev, steps=None, warmup=None):
    """64 independent three-material tool scenes on 64^3 grids (particle counts
    log-uniform in [1e4, 1.5e5], about 3.3M in all) stepped by one launch per
    stage: 100 steps forward + adjoint of the per-scene position loss w.r.t.
    every scene's actions, checkpoint every 20, CUDA graphs, autotuned
    launch shapes."""
    import torch

    import scenes
    from paper_2303_02346_gb300 import binding as B
    from paper_2303_02346_gb300.simulator import Simulator
    steps = args.steps if steps is None else steps
    warmup = args.warmup if warmup is None else warmup
    sc = scenes.batched_scenes()
    T, N, S = sc.n_steps, sc.n_particles, sc.n_scenes
    sim = Simulator(sc, checkpoint_every=20, max_steps=T, device=dev)
    h = sim.h
    x0 = torch.tensor(sc.x, dtype=torch.float32, device=dev)
    v0 = torch.tensor(sc.v, dtype=torch.float32, device=dev)
    mat = torch.tensor(sc.mat, dtype=torch.uint8, device=dev)
    pose0 = torch.tensor(sc.tool_pose0, dtype=torch.float32, device=dev)
    acts = torch.tensor(sc.tool_actions, dtype=torch.float32, device=dev)
    tgt = sc.loss["target"]
    ga = torch.empty(S, acts.shape[1], 6, dtype=torch.float32, device=dev)
    stream = torch.cuda.current_stream(dev)

    def trajectory(ev=None):
        B.sim_set_particles(h, -1, x0, v0, mat)
        B.sim_set_tool(h, -1, pose0, acts, acts.shape[1])
        if ev is not None:
            ev[0].record(stream)
        B.sim_step(h, T)
        if ev is not None:
            ev[1].record(stream)
        B.sim_position_loss(h, -1, tgt, 1.0, n_out=S)
        B.sim_backward(h, None, None, ga)

    B.sim_set_particles(h, -1, x0, v0, mat)
    B.sim_set_tool(h, -1, pose0, acts, acts.shape[1])
    tuning = B.sim_autotune(h, 20)
    for _ in range(max(warmup, 1)):
        trajectory()
    torch.cuda.synchronize()
    tot, fwd = [], []
    for _ in range(max(steps, 1)):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(4)]
        e[0].record(stream)
        trajectory((e[1], e[2]))
        e[3].record(stream)
        torch.cuda.synchronize()
        tot.append(e[0].elapsed_time(e[3]))
        fwd.append(e[1].elapsed_time(e[2]))
    ms, fms = statistics.median(tot), statistics.median(fwd)
    sim.close()
    return {
        "workload": f"{S} three-material tool scenes on 64^3 (counts log-uniform in [1e4, 1.5e5]), "
                    f"{N} particles, {T} steps forward + adjoint of a per-scene position loss, checkpoint every 20",
        "particles": N, "scenes": S, "steps": T, "ms_per_trajectory": round(ms, 3),
        "value": round(N * T / (ms / 1e3), 1), "unit": UNIT,
        "fwd": {"value": round(N * T / (fms / 1e3), 1), "ms": round(fms, 3)},
        "launch": {"scatter_threads": tuning[0], "gather_threads": tuning[1], "grid_blocks_per_cta": tuning[2],
                   "fused_adjoint": bool(tuning[4]), "persistent_forward": bool(tuning[5]),
                   "staged_gather": bool(tuning[6]), "scatter_ctas_per_sm": tuning[7], "cuda_graphs": True,
                   "autotuned": True},
    }


def run_rigid(args, dev):
    """The bench scene (200k particles, 128^3, box tool, 200 steps forward +
    grid-mass loss adjoint, checkpoint every 20) with its 40k-particle sand
    block made a rigid body (Sec. 3.2 "Rigid body"); the same scene with the
    sand block is timed beside it on the same handle shapes (CUDA events,
    median of the timed trajectories)."""
    import torch

    import scenes
    from paper_2303_02346_gb300 import binding as B
    from paper_2303_02346_gb300.simulator import Simulator
    out = {}
    for name in ("three_material", "rigid"):
        sc = scenes.multi_material(scale=args.scale)
        if name == "rigid":
            sc.materials[2] = scenes.rigid_material(sc.materials[2].volume)
        T, N = sc.n_steps, sc.n_particles
        sim = Simulator(sc, checkpoint_every=20, max_steps=T, device=dev)
        h = sim.h
        x0 = torch.tensor(sc.x, dtype=torch.float32, device=dev)
        v0 = torch.tensor(sc.v, dtype=torch.float32, device=dev)
        mat = torch.tensor(sc.mat, dtype=torch.uint8, device=dev)
        pose0 = torch.tensor(sc.tool_pose0, dtype=torch.float32, device=dev)
        acts = torch.tensor(sc.tool_actions, dtype=torch.float32, device=dev)
        tm = torch.tensor(sc.loss["target_mass"], dtype=torch.float32, device=dev)
        td = torch.tensor(sc.loss["target_dist"], dtype=torch.float32, device=dev)
        M = float(sc.loss["total_mass"])
        ga = torch.empty(1, acts.shape[1], 6, dtype=torch.float32, device=dev)
        stream = torch.cuda.current_stream(dev)

        def trajectory(ev=None):
            B.sim_set_particles(h, -1, x0, v0, mat)
            B.sim_set_tool(h, -1, pose0, acts, acts.shape[1])
            if ev is not None:
                ev[0].record(stream)
            B.sim_step(h, T)
            if ev is not None:
                ev[1].record(stream)
            B.sim_grid_mass_loss(h, 0, tm, td, M)
            B.sim_backward(h, None, None, ga)

        sim.reset()
        tuning = B.sim_autotune(h, 20)
        for _ in range(max(args.warmup, 1)):
            trajectory()
        torch.cuda.synchronize()
        tot, fwd = [], []
        for _ in range(max(args.steps, 1)):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(4)]
            e[0].record(stream)
            trajectory((e[1], e[2]))
            e[3].record(stream)
            torch.cuda.synchronize()
            tot.append(e[0].elapsed_time(e[3]))
            fwd.append(e[1].elapsed_time(e[2]))
        ms, fms = statistics.median(tot), statistics.median(fwd)
        # per-stage event timings of one more trajectory (serial: no graphs, no overlap)
        B.sim_profile_enable(h, 1)
        trajectory()
        prof = B.sim_profile_read(h)
        B.sim_profile_enable(h, 0)
        sim.close()
        out[name] = {"ms_per_trajectory": round(ms, 3), "fwd_ms": round(fms, 3),
                     "value": round(N * T / (ms / 1e3), 1), "fwd_value": round(N * T / (fms / 1e3), 1),
                     "unit": UNIT, "tuning": list(tuning),
                     "stages_us_avg": {k: round(1e3 * v[0] / max(v[1], 1), 2) for k, v in prof.items()}}
    out["workload"] = ("bench scene (200k particles, 128^3, box tool, 200 steps + grid-mass loss adjoint) "
                       "with the 40k-particle sand block as a particle-represented rigid body")
    return out


# ----------------------------------------------------------------------------
# learned surrogate
# ----------------------------------------------------------------------------
SUR_N = 64
SUR_CONV_FLOPS_PER_NODE = 2 * 27 * 32 * 32  # one 3x3x3 conv, 32 -> 32 channels


def _timed(stream, fn, reps):
    import torch
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(reps)]
    for a, b in ev:
        a.record(stream)
        fn()
        b.record(stream)
    torch.cuda.synchronize()
    return [a.elapsed_time(b) for a, b in ev]


def run_sharing(args, dev, reps=10):
    """Gradient sharing and the attraction loss (Sec. 5.1) on the bench scene
    after 20 steps: each call bins the particles by cell at their current
    positions and sums over the neighbours within 0.8 dx (CUDA events)."""
    import torch

    import scenes
    from paper_2303_02346_gb300 import binding as B
    from paper_2303_02346_gb300.simulator import Simulator
    sc = scenes.multi_material(scale=args.scale)
    sim = Simulator(sc, checkpoint_every=20, max_steps=20)
    sim.reset()
    sim.step(20)
    N = sc.n_particles
    g = torch.Generator(device=dev).manual_seed(0)
    ell = torch.rand(N, generator=g, device=dev)
    grad = torch.randn(N, 3, generator=g, device=dev)
    out = torch.empty_like(grad)
    h, tau = 0.8 / sc.grid_n, 0.5
    stream = torch.cuda.current_stream(dev)

    def timed(fn):
        fn()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(reps):
            fn()
        e1.record(stream)
        torch.cuda.synchronize()
        return e0.elapsed_time(e1) / reps

    t_att = timed(lambda: B.sim_attraction_loss(sim.h, -1, ell, h, tau, 1.0))
    t_share = timed(lambda: B.sim_share_gradients(sim.h, -1, ell, h, tau, grad, out))
    sim.close()
    return {"what": f"{N} particles, radius 0.8 dx, bin by cell + neighbour sum per call (host-synchronous)",
            "attraction_ms": round(t_att, 3), "attraction_particles_per_s": round(N / (t_att / 1e3), 1),
            "share_ms": round(t_share, 3), "share_particles_per_s": round(N / (t_share / 1e3), 1)}


def run_gas(args, dev, n=256, T=8, reps=3):
    """Gas solver (Sec. 3.2, Stam 1999) on a 256^3 box with a block obstacle:
    steps/s forward and forward + adjoint (CUDA events around whole
    trajectories, graphs captured during an untimed warm-up), and the HBM
    roofline of a pass of two Jacobi sweeps, timed as the marginal step time
    between 20 and 60 sweeps (13 algorithmic bytes per cell and pass: p, the
    right-hand side and the solid byte read, p written)."""
    import numpy as np
    import torch

    from paper_2303_02346_gb300.gas import GasSolver
    solid = np.zeros((n, n, n), dtype=np.uint8)
    solid[0, :, :] = solid[-1, :, :] = solid[:, 0, :] = solid[:, -1, :] = solid[:, :, 0] = solid[:, :, -1] = 1
    c = n // 2
    solid[c - n // 8:c + n // 8, c:c + n // 16, c - n // 8:c + n // 8] = 1
    g = torch.Generator(device=dev).manual_seed(0)
    fl = torch.as_tensor(solid == 0, device=dev)
    u0 = (0.5 * torch.randn(3, n, n, n, generator=g, device=dev)) * fl
    d0 = torch.rand(n, n, n, generator=g, device=dev) * fl
    wu = torch.randn(3, n, n, n, generator=g, device=dev)
    stream = torch.cuda.current_stream(dev)

    def timed(fn):
        fn()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(reps):
            fn()
        e1.record(stream)
        torch.cuda.synchronize()
        return e0.elapsed_time(e1) / reps

    res = {}
    for K in (20, 60):
        gs = GasSolver(n, 0.002, 4.0, K, T, solid, device=dev)

        def fwd():
            gs.set_state(u0, d0)
            gs.step(T)

        def fwd_adj():
            fwd()
            gs.add_grad(wu, None)
            gs.backward()

        res[K] = (timed(fwd), timed(fwd_adj), gs.launches())
        gs.close()
        del gs
    K = 60
    t_fwd, t_all, _ = res[K]
    sweep_ms = (res[60][0] - res[20][0]) / (T * 40)
    launch_ms, launch_bytes = 2 * sweep_ms, 13 * n ** 3  # two sweeps a launch, every field moved once
    peak, src = load_peaks()
    achieved = launch_bytes / (launch_ms / 1e3) / 1e9
    cells = float(n) ** 3 * T
    return {"workload": f"{n}^3 cells, box walls and a block obstacle, {T} steps, {K} damped Jacobi sweeps per "
                        "projection, forward + adjoint of a linear loss on the final velocity",
            "fwd_ms_per_step": round(t_fwd / T, 3), "fwd_adj_ms_per_step": round(t_all / T, 3),
            "fwd_cell_steps_per_s": round(cells / (t_fwd / 1e3), 1),
            "fwd_adj_cell_steps_per_s": round(cells / (t_all / 1e3), 1),
            "roofline": {"bound": "hbm", "kernel": "jacobi2_kernel", "achieved": round(achieved, 1),
                         "peak": peak, "peak_source": src, "unit": "GB/s", "frac": round(achieved / peak, 4),
                         "traffic": profiled_traffic("gas_jacobi2"),
                         "algorithmic_bytes_per_launch": launch_bytes, "avg_launch_ms": round(launch_ms, 5),
                         "timing": "marginal step time of two sweeps, 60 against 20 sweeps"}}


def run_surrogate_quick(args, dev):
    """Speed of the conv surrogate on 64^3 frames (batch 8, seeded random
    weights and frames): inference and training frames/s and the tensor-core
    roofline of the convolution kernel (CUDA events per launch)."""
    import torch

    from paper_2303_02346_gb300.surrogate import Surrogate, init_params
    n, bt = SUR_N, 8
    sur = Surrogate(n, 1.0, 1.0, max_batch=bt, device=dev)
    sur.set_params(init_params(0))
    g = torch.Generator(device=dev).manual_seed(0)
    frames = torch.randn(2 * bt, n ** 3, 8, generator=g, device=dev).to(torch.bfloat16).view(torch.int16)
    idx = torch.arange(bt, dtype=torch.int32, device=dev)
    tgt = idx + bt
    pred = torch.empty(bt, n ** 3, 3, device=dev)
    stream = torch.cuda.current_stream(dev)
    from paper_2303_02346_gb300 import binding as B
    infer = lambda: B.sur_predict(sur.h, bt, frames, idx, pred)
    train = lambda: sur.train_step(frames, idx, tgt, 1e-5)
    for _ in range(3):
        infer()
        train()
    if args.profile_only:
        for _ in range(args.steps):
            infer()
            train()
        torch.cuda.synchronize()
        sur.close()
        return None
    l0 = B.sur_kernel_launches(sur.h)
    t_inf = _timed(stream, infer, max(args.steps, 3))
    per_infer = (B.sur_kernel_launches(sur.h) - l0) / max(args.steps, 3)
    t_train = _timed(stream, train, max(args.steps, 3))
    sur.profile(True)
    for _ in range(max(args.steps, 3)):
        infer()
    prof_inf = sur.profile_read()
    sur.profile(False)
    sur.profile(True)
    for _ in range(max(args.steps, 3)):
        train()
    prof_train = sur.profile_read()
    sur.profile(False)
    conv_ms = prof_inf["sur_conv3_umma"][0] / prof_inf["sur_conv3_umma"][1]
    flops = SUR_CONV_FLOPS_PER_NODE * bt * n ** 3
    peak, src = load_tensor_peak()
    achieved = flops / (conv_ms / 1e3) / 1e12
    inf_ms = statistics.median(t_inf)
    tr_ms = statistics.median(t_train)
    out = {
        "workload": f"conv surrogate, {bt} frames of {n}^3 x 8 channels, 4 residual blocks, 32 channels, BF16",
        "inference_frames_per_s": round(bt / (inf_ms / 1e3), 1), "inference_ms_per_batch": round(inf_ms, 3),
        "train_frames_per_s": round(bt / (tr_ms / 1e3), 1), "train_ms_per_step": round(tr_ms, 3),
        "kernel_launches_per_inference": per_infer,
        "roofline": {"bound": "tensor", "kernel": "sur_conv3_umma", "achieved": round(achieved, 1),
                     "peak": peak, "peak_source": src + " (burst)", "unit": "TFLOP/s",
                     "frac": round(achieved / peak, 4), "traffic": profiled_traffic("sur_conv3_umma"),
                     "algorithmic_flops_per_launch": flops, "avg_launch_ms": round(conv_ms, 5)},
        "kernels_inference": {k: {"ms_avg": round(v[0] / max(v[1], 1), 5), "launches": v[1]}
                              for k, v in prof_inf.items()},
        "kernels_train": {k: {"ms_avg": round(v[0] / max(v[1], 1), 5), "launches": v[1]}
                          for k, v in prof_train.items()},
    }
    sur.close()
    return out


def run_surrogate(args, build=True):
    """Frames from 64-scene rollouts (three-material tool scenes on 64^3),
    training, held-out relative L2 error, error gate with simulation fallback,
    and speed against the simulation."""
    import numpy as np
    import torch

    import scenes
    from paper_2303_02346_gb300 import build as b
    from paper_2303_02346_gb300 import surrogate as SG
    if build:
        b.build()
    dev = torch.device("cuda", 0)
    R, T, H = args.sur_rollouts, args.sur_rollout_steps, 10
    scs = [scenes.batched_scenes(seed=5 + r, n_steps=T) for r in range(R)]
    S = scs[0].n_scenes
    m_ref, v_ref = SG.frame_scales(scs[0])
    sur = SG.Surrogate(SUR_N, m_ref, v_ref, max_batch=args.sur_batch, device=dev)
    sur.set_params(SG.init_params(5))
    frames = sur.empty_frames(R * (T + 1) * S)
    sim_ms = []
    idx_all, tgt_all, scene_all = [], [], []
    t0 = time.perf_counter()
    for r, sc in enumerate(scs):
        _, i, t, s = SG.generate_frames(sur, sc, T, H, out=frames, first=r * (T + 1) * S, timer=sim_ms)
        idx_all.append(i)
        tgt_all.append(t)
        scene_all.append(s)
    gen_s = time.perf_counter() - t0
    idx, tgt, scn = np.concatenate(idx_all), np.concatenate(tgt_all), np.concatenate(scene_all)
    val = scn >= int(round(0.9 * S))  # the last 10% of each rollout's scenes are held out
    tr_i, tr_t, va_i, va_t = idx[~val], tgt[~val], idx[val], tgt[val]
    # identity baseline: predict the current momentum
    f = frames.view(torch.bfloat16)
    ident = []
    for k in range(0, len(va_i), 64):
        a = f[torch.as_tensor(va_i[k:k + 64], device=dev)][..., 1:4].float()
        c = f[torch.as_tensor(va_t[k:k + 64], device=dev)][..., 1:4].float()
        ident.append((torch.linalg.norm((a - c).reshape(a.shape[0], -1), dim=1) /
                      torch.linalg.norm(c.reshape(c.shape[0], -1), dim=1)).cpu().numpy())
    ident = np.concatenate(ident)
    err0 = SG.evaluate(sur, frames, va_i, va_t)
    t1 = time.perf_counter()
    hist = SG.train(sur, frames, tr_i, tr_t, args.sur_train_steps, args.sur_batch, args.sur_lr, seed=5)
    torch.cuda.synchronize()
    train_s = time.perf_counter() - t1
    err = SG.evaluate(sur, frames, va_i, va_t)
    err_tr = SG.evaluate(sur, frames, tr_i[:len(va_i)], tr_t[:len(va_i)])
    # speed: one prediction of a 64-scene batch vs the 10 simulation steps it replaces
    stream = torch.cuda.current_stream(dev)
    sel = torch.as_tensor(va_i[:args.sur_batch], dtype=torch.int32, device=dev)
    pred = torch.empty(args.sur_batch, SUR_N ** 3, 3, device=dev)
    from paper_2303_02346_gb300 import binding as B
    for _ in range(3):
        B.sur_predict(sur.h, args.sur_batch, frames, sel, pred)
    t_inf = statistics.median(_timed(stream, lambda: B.sur_predict(sur.h, args.sur_batch, frames, sel, pred), 10))
    ms_per_frame = t_inf / args.sur_batch
    mpm_ms_per_step = float(np.sum(sim_ms)) / (R * T)          # all S scenes, one step
    mpm_ms_per_scene_10 = mpm_ms_per_step * H / S              # one scene, 10 steps
    bound = args.sur_bound
    frac_fallback = float(np.mean(err > bound))
    # gradients against the simulation: dL/dv at step 40 of the last rollout
    held = np.arange(S) >= int(round(0.9 * S))
    grad_cmp = {}
    for field in ("smooth", "white"):
        cg = SG.compare_gradients(sur, scs[-1], 40, H, seed=1, field=field)
        grad_cmp[field] = {
            "rel_l2_median": float(np.median(cg["rel_l2"][held])),
            "cosine_median": float(np.median(cg["cosine"][held])),
            "no_change_rel_l2_median": float(np.median(cg["identity_rel_l2"][held])),
            "no_change_cosine_median": float(np.median(cg["identity_cosine"][held])),
            "all_scenes_cosine_median": float(np.median(cg["cosine"]))}
    return {
        "workload": f"conv surrogate on {SUR_N}^3 frames from {R} rollouts x {S} three-material tool scenes "
                    f"x {T + 1} steps (batched-scene generator, seeds 5..{4 + R}); target = grid momentum "
                    f"{H} steps ahead; scenes >= {int(round(0.9 * S))} of each rollout held out",
        "frames": int(frames.shape[0]), "pairs_train": int(len(tr_i)), "pairs_val": int(len(va_i)),
        "frame_bytes": int(frames.numel() * 2), "generate_s": round(gen_s, 2),
        "train_steps": args.sur_train_steps, "batch": args.sur_batch, "lr": args.sur_lr,
        "train_s": round(train_s, 2),
        "train_frames_per_s": round(args.sur_train_steps * args.sur_batch / train_s, 1),
        "loss_first_last": [float(np.mean(hist[:20])), float(np.mean(hist[-20:]))],
        "val_rel_l2": {"mean": float(np.mean(err)), "median": float(np.median(err)),
                       "p90": float(np.quantile(err, 0.9)), "max": float(np.max(err))},
        "val_rel_l2_untrained": float(np.mean(err0)),
        "train_rel_l2_mean": float(np.mean(err_tr)),
        "identity_rel_l2": {"mean": float(np.mean(ident)), "median": float(np.median(ident))},
        "gradients_vs_simulation": dict(
            what=f"dL/dv at step 40 of the last rollout for L = <w, momentum {H} steps later>; surrogate "
                 f"(features -> network -> adjoint) against the simulation's adjoint on held-out scenes; w = "
                 f"smooth (4 plane waves per component, wavelength >= {SUR_N // 3} nodes) or white noise",
            **grad_cmp),
        "gate": {"bound": bound, "fallback_fraction": round(frac_fallback, 4),
                 "fallback_fraction_at": {str(b_): round(float(np.mean(err > b_)), 4)
                                          for b_ in (0.02, 0.05, 0.1, 0.2, 0.3)},
                 "identity_fallback_fraction": round(float(np.mean(ident > bound)), 4)},
        "speed": {"surrogate_ms_per_frame": round(ms_per_frame, 4),
                  "simulation_ms_per_scene_10_steps": round(mpm_ms_per_scene_10, 4),
                  "simulation_ms_per_batched_step_64_scenes": round(mpm_ms_per_step, 4),
                  "speedup_vs_simulation": round(mpm_ms_per_scene_10 / ms_per_frame, 3),
                  "speedup_with_fallback": round(mpm_ms_per_scene_10 /
                                                 (ms_per_frame + frac_fallback * mpm_ms_per_scene_10), 3)},
    }


# ----------------------------------------------------------------------------
# oracle (CPU) legs
# ----------------------------------------------------------------------------
def oracle_sample(n_steps=1, scale=1.0):
    """Time the FP64 oracle (as it stands) on the bench workload (the dam-break
    scene): n_steps forward MPM steps + autograd adjoint of the final-position
    loss w.r.t. the initial positions. Returns (particle-steps/s, seconds,
    threads, particles)."""
    import torch

    import scenes
    from oracle import mpm as omp
    sc = scenes.dam_break(scale=scale)
    x0 = torch.tensor(sc.x, dtype=torch.float64, requires_grad=True)
    t0 = time.perf_counter()
    x, v, C, F = omp.rollout(sc, n_steps=n_steps, x0=x0)
    L = omp.scene_loss(sc, x)
    L.backward()
    dt = time.perf_counter() - t0
    return sc.n_particles * n_steps / dt, dt, torch.get_num_threads(), sc.n_particles


def run_reference(args, rank):
    if rank != 0:
        return None
    vals, secs = [], []
    for i in range(args.warmup + args.steps):
        v, dt, threads, N = oracle_sample(1, args.scale)
        if i >= args.warmup:
            vals.append(v)
            secs.append(dt)
    value = len(vals) / sum(secs) * N
    sample = f"{N} particles x 1 MPM step forward + autograd adjoint per bench step (FP64 oracle)"
    return {
        "impl": "reference", "metric": METRIC, "value": round(value, 1), "unit": UNIT,
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": round(1e3 * sum(secs) / len(secs), 1), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": WORKLOAD, "particles": N},
        "cpu_baseline": {"value": round(value, 1), "unit": UNIT, "cores": threads, "kind": "oracle",
                         "sample": sample},
        "e2e": {"value": round(value, 1), "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }


def main():
    args = parse()
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    if args.impl == "reference":
        out = run_reference(args, rank)
        if out is not None:
            print(json.dumps(out), flush=True)
        return
    if args.workload in ("dam_break", "multi_material"):
        if rank == 0:
            import torch

            import scenes
            from paper_2303_02346_gb300 import build as b
            b.build()
            dev = torch.device("cuda", 0)
            # smaller copies (grid, horizon, checkpoint interval) serve profiler captures
            kw = {}
            if args.grid_n:
                kw["grid_n"] = args.grid_n
            if args.horizon:
                kw["n_steps"] = args.horizon
            if args.checkpoint_every:
                kw["checkpoint_every"] = args.checkpoint_every
            sc = scenes.dam_break(scale=args.scale, **kw) if args.workload == "dam_break" else \
                scenes.multi_material(scale=args.scale, **kw)
            label = args.workload if not kw and args.scale == 1.0 else sc.name
            out = run_trajectory(args, sc, dev, 0, 1, args.steps, args.warmup, label=label)
            if out is not None:
                print(json.dumps(out), flush=True)
        return
    if args.workload == "surrogate":
        if rank == 0:
            print(json.dumps(run_surrogate(args)), flush=True)
        return
    if args.workload == "batched":
        if rank == 0:
            import torch
            from paper_2303_02346_gb300 import build as b
            b.build()
            print(json.dumps(run_batched(args, torch.device("cuda", 0))), flush=True)
        return
    if args.workload == "rigid":
        if rank == 0:
            import torch
            from paper_2303_02346_gb300 import build as b
            b.build()
            print(json.dumps(run_rigid(args, torch.device("cuda", 0))), flush=True)
        return
    if args.workload == "gas":
        if rank == 0:
            import torch
            from paper_2303_02346_gb300 import build as b
            b.build()
            print(json.dumps(run_gas(args, torch.device("cuda", 0))), flush=True)
        return
    if args.workload == "surrogate_speed":
        if rank == 0:
            import torch
            from paper_2303_02346_gb300 import build as b
            b.build()
            out = run_surrogate_quick(args, torch.device("cuda", 0))
            if out is not None:
                print(json.dumps(out), flush=True)
        return
    import torch
    if world > 1:
        torch.cuda.set_device(local_rank)
        torch.distributed.init_process_group("nccl", device_id=torch.device("cuda", local_rank))
    out = run_ours(args, rank, world, local_rank)
    if out is not None and rank == 0 and not args.no_cpu_baseline:
        v, dt, threads, N = oracle_sample(2, args.scale)
        out["cpu_baseline"] = {"value": round(v, 1), "unit": UNIT, "cores": threads, "kind": "oracle",
                               "sample": f"dam-break scene, {N} particles x 2 MPM steps forward + autograd "
                                         f"adjoint of the final-position loss ({dt:.1f} s, FP64 oracle on the "
                                         f"host cores)"}
    if out is not None and rank == 0:
        print(json.dumps(out), flush=True)
    if world > 1:
        torch.distributed.destroy_process_group()


if __name__ == "__main__":
    main()
