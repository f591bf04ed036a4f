#!/usr/bin/env python3
"""Benchmark: Gcell/s of one full time step of the PLIC / split-VOF /
consistent-energy hot path (three direction sweeps + phase-change shift +
FP64 sums) on the 256^3 vapour-bubble growth workload (Sec. 4.4 shape:
vapour sphere R0 = 0.1 in superheated water, erf thermal layer of
thickness 0.02, Ja = 0.5, radial liquid velocity, mass-flux-driven shift).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl gpu|reference]

One rank per GPU (torchrun for N > 1); every rank advances its own replica
of the workload (weak scaling, no collective on the data path); the timed
region is bracketed by a barrier and a device synchronise, the time is the
max over ranks, and rank 0 prints one JSON line.

--impl reference times the FP64 CPU oracle (test infrastructure) on the
host cores on a bounded sample of the same workload.
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "Gcell/s per 3-sweep PLIC+energy advection step; % of HBM roofline"
UNIT = "Gcell/s"
N_CELLS = 256
# Algorithmic bytes per cell of one time step of the FP64 form: each sweep
# reads c, e, the face velocity of its axis, the frozen Theta (8 B each) and
# cc (1 B) and writes c, e (49 B); the first sweep also writes Theta and cc
# (9 B); the shift reads c, e and the per-cell shift dd and writes c, e
# (40 B): 3 x 49 + 9 + 40 = 196 B.  (The kernels move less: Theta is
# written only for cells that change, and quiet tiles are skipped.)
SWEEP_BYTES_PER_CELL = 8 + 8 + 8 + 8 + 1 + 8 + 8
STEP_BYTES_PER_CELL = 3 * SWEEP_BYTES_PER_CELL + 9 + 40
# nominal HBM3e bandwidth of one GB300 (the roofline itself uses the measured copy rate)
HBM_NOMINAL_GBS = 7900.0


def max_over_ranks(x, world, device):
    """The largest of the ranks' values of x (every rank gets it)."""
    if world <= 1:
        return float(x)
    import torch
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_throughput(cells, steps, world, seconds):
    """Whole-job Gcell/s: every rank advances its own replica (weak scaling),
    timed by the slowest rank."""
    return cells * steps * world / seconds / 1e9


def dist_env():
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return rank, world, local


class ClockSampler:
    """nvidia-smi clocks / throttle reasons sampled during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "100"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except (OSError, FileNotFoundError):
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.thread.join(timeout=2)
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                mx = float(parts[2])
            except ValueError:
                continue
            for nm, val in zip(names, parts[5:9]):
                if val.lower() == "active":
                    reasons.add(nm)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": mx, "reasons": sorted(reasons),
                "samples": len(sm)}


def measured_peak_gbs():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return float(json.load(f)["hbm_gbs"]), "measured"
    except (OSError, KeyError, ValueError):
        return 6800.0, "fallback"


# FP64 work of k_walk per face and cell (pure, fused multiply-adds count two
# flop): T = e / C_p 1, the difference of T 1, a = u lambda 1, T_f = v0 +
# correction / 6 2, G = (T_f C_p) a 2, Theta = C_p T 1, e' = (e + (G_l - Theta
# a_l)) - (G_r - Theta a_r) 6: 14 flop in 13 instructions.  The WENO5
# correction itself (64 of the method's 78 flop) runs in pairs of FP32 numbers.
FACE_FLOP, FACE_INSTR = 14, 13
FACE_SOURCES = ("paper_2001_03477_gb300/csrc/vof_fused.cu", "paper_2001_03477_gb300/csrc/vof_sweep.cuh",
                "paper_2001_03477_gb300/csrc/vof_df.cuh", "paper_2001_03477_gb300/csrc/vof_device.cuh")


def sources_sha1(paths):
    import hashlib
    h = hashlib.sha1()
    for p in paths:
        with open(os.path.join(ROOT, p), "rb") as f:
            h.update(f.read())
    return h.hexdigest()


def faces_traffic_from_profile():
    """DRAM bytes per launch of the step's face kernel (k_walk) from the
    committed ncu summary, if it was taken on the current sources of that
    kernel; None otherwise."""
    path = os.path.join(ROOT, "profiles", "k_faces_traffic.json.txt")
    try:
        with open(path) as f:
            d = json.load(f)
        if d.get("sources_sha1") != sources_sha1(FACE_SOURCES):
            return None
        return float(d["dram_bytes_per_launch"])
    except (OSError, KeyError, ValueError):
        return None


def fp64_peak_tflops(sm_max_mhz):
    """FP64 peak derived from unit counts and clock: 152 SMs x 2 FP64 FMA
    lanes-ops per SM per clock x 2 flop, at the maximum SM clock seen."""
    mhz = sm_max_mhz if sm_max_mhz else 2070.0
    return 152 * 2 * 2 * mhz * 1e6 / 1e12


def load_workload():
    from paper_2001_03477_gb300 import workloads as W
    return W.bubble_growth(n=N_CELLS, nsub=8)


def run_gpu(args):
    import torch
    import torch.distributed as dist
    import paper_2001_03477_gb300 as P
    from paper_2001_03477_gb300 import build

    rank, world, local = dist_env()
    if world > 1:
        dist.init_process_group("nccl", init_method="env://")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if rank == 0 or not os.path.exists(P.LIB_PATH):
        build.build()
    if world > 1:
        dist.barrier()

    wl = load_workload()
    g = P.Grid(wl.shape[2], wl.shape[1], wl.shape[0], wl.bc, wl.h, wl.Cp_l, wl.Cp_g, wl.T_sat)
    c0 = torch.from_numpy(wl.c).to(dev)
    e0 = torch.from_numpy(wl.e).to(dev)
    u = torch.from_numpy(wl.u).to(dev)
    v = torch.from_numpy(wl.v).to(dev)
    w = torch.from_numpy(wl.w).to(dev)
    c, e = c0.clone(), e0.clone()
    # the Step-2 shift as a per-cell array (the mass-flux-driven interface
    # shift of the workload, equal in every cell here)
    dd = torch.full_like(c0, wl.dd_uniform)
    st = P.Stepper(g, device=dev)
    stream = torch.cuda.current_stream(dev)

    def barrier():
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize(dev)

    # ---- device-resident timed region --------------------------------------
    for s in range(args.warmup):
        st.step(c, e, u, v, w, wl.dt, s, dd=dd)
    barrier()
    sampler = ClockSampler(local) if rank == 0 else None
    if sampler:
        sampler.start()
        time.sleep(0.3)
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    barrier()
    ev0.record(stream)
    for s in range(args.steps):
        st.step(c, e, u, v, w, wl.dt, args.warmup + s, dd=dd)
    ev1.record(stream)
    barrier()
    clocks = sampler.stop() if sampler else None
    ms = ev0.elapsed_time(ev1)
    ms = max_over_ranks(ms, world, dev)
    sums = st.sums.cpu().numpy()
    cells = wl.cells
    value = job_throughput(cells, args.steps, world, ms * 1e-3)

    # ---- per-launch durations of the same step ----------------------------
    # the library records a CUDA event on the launching stream after each of
    # its launches (vof_profile_begin/end); durations are per step, averaged
    # over `reps` steps run right after the timed region
    reps = max(3, min(args.steps, 20))
    barrier()
    P.vof_profile_begin(stream)
    for r in range(reps):
        st.step(c, e, u, v, w, wl.dt, args.warmup + args.steps + r, dd=dd)
    launches = P.vof_profile_end()
    barrier()
    kern_ms = {}
    for name, t in launches:
        kern_ms[name] = kern_ms.get(name, 0.0) + t / reps
    kernels_per_step = sum(1 for name, _ in launches if "memset" not in name) // reps
    peak, peak_kind = measured_peak_gbs()
    counts = P.vof_step_work_counts(g, st.workspace, stream)
    # the dominant kernel: k_walk (its three launches take the largest share
    # of the step); bound by the instructions of the faces it evaluates, FP64
    # and others
    faces_ms = sum(kern_ms.get(f"sweep_{a}.walk", 0.0) for a in "xyz")
    faces_per_step = sum(counts["faces"])
    step_ms_prof = sum(kern_ms.values())
    fp64_achieved = FACE_FLOP * faces_per_step / (faces_ms * 1e-3) / 1e12 if faces_ms > 0 else 0.0
    traffic = faces_traffic_from_profile()
    fp64 = fp64_rate(P, dev, stream) if rank == 0 else None
    fp64_peak = fp64["dfma_tflops"] if fp64 else fp64_peak_tflops(clocks["sm_max_mhz"] if clocks else None)

    # ---- the mass transfer rate (Sec. 3.2) on the same workload -------------
    mt = None if args.step_only else mass_transfer_measure(P, g, wl, c0, e0, stream, barrier)
    # ---- the step with Li's Lagrangian-explicit sweeps (the other Step 1) ----
    le = None if args.step_only else scheme_le_measure(P, wl, c0, e0, u, v, w, stream, barrier,
                                                       steps=min(args.steps, 100))

    # ---- end to end through the public API with host buffers ---------------
    # each step the face velocities of the liquid (produced by the flow
    # solver on the host) are copied in from pinned memory, the step runs,
    # and its sums are read back on the host.  The copies run on their own
    # stream into two alternating device buffers: step s+1's velocities come
    # in while step s computes, and step s's sums are read once step s+1 is
    # queued.
    uh = torch.from_numpy(wl.u).pin_memory()
    vh = torch.from_numpy(wl.v).pin_memory()
    wh = torch.from_numpy(wl.w).pin_memory()
    host_in = (uh, vh, wh)
    bufs = [(u, v, w), tuple(torch.empty_like(t) for t in (u, v, w))]
    sums_h = [torch.empty(P.VOF_NSUMS, dtype=torch.float64).pin_memory() for _ in range(2)]
    copy_stream = torch.cuda.Stream(dev)
    ready = [torch.cuda.Event(), torch.cuda.Event()]   # velocities of buffer b copied in
    free = [torch.cuda.Event(), torch.cuda.Event()]    # the step reading buffer b has run
    got = [torch.cuda.Event(), torch.cuda.Event()]     # sums of the step of buffer b copied out
    for b in range(2):
        free[b].record(stream)

    def issue_copy(b):
        copy_stream.wait_event(free[b])
        with torch.cuda.stream(copy_stream):
            for dst, src in zip(bufs[b], host_in):
                dst.copy_(src, non_blocking=True)
        ready[b].record(copy_stream)

    def e2e_run(nsteps):
        total = 0.0
        issue_copy(0)
        for s_ in range(nsteps):
            b = s_ % 2
            if s_ + 1 < nsteps:
                issue_copy(1 - b)
            stream.wait_event(ready[b])
            st.step(c, e, *bufs[b], wl.dt, s_, dd=dd)
            free[b].record(stream)
            sums_h[b].copy_(st.sums, non_blocking=True)
            got[b].record(stream)
            if s_ >= 1:
                got[1 - b].synchronize()
                total += float(sums_h[1 - b][0])
        got[(nsteps - 1) % 2].synchronize()
        return total + float(sums_h[(nsteps - 1) % 2][0])

    c.copy_(c0); e.copy_(e0)
    e2e_steps = max(3, min(args.steps, 100))
    e2e_run(2)
    barrier()
    t0 = time.perf_counter()
    e2e_run(e2e_steps)
    barrier()
    e2e_s = time.perf_counter() - t0
    e2e_s = max_over_ranks(e2e_s, world, dev)
    e2e_value = job_throughput(cells, e2e_steps, world, e2e_s)
    h2d = (wl.u.nbytes + wl.v.nbytes + wl.w.nbytes)

    if rank == 0:
        cpu = cpu_baseline() if world == 1 and not args.no_cpu_baseline else None
        del c, e, c0, e0, u, v, w, st
        torch.cuda.empty_cache()
        pform = (precision_form(dev, fp64_peak=fp64_peak, hbm_peak=peak)
                 if world == 1 and not (args.no_precision_form or args.step_only) else None)
        learned = (learned_form(dev, fp64_peak=fp64_peak)
                   if world == 1 and not (args.no_learned_form or args.step_only) else None)
        torch.cuda.empty_cache()
        batched = (batched_form(dev) if world == 1 and not (args.no_batched_form or args.step_only) else None)
        out = {
            "metric": METRIC, "value": round(value, 4), "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": f"bubble-growth {N_CELLS}^3 (vapour R0=0.1, erf layer 0.02, Ja=0.5, water/steam "
                                   f"Cp ratio {wl.Cp_l / wl.Cp_g:.1f}, radial u_l, uniform shift {wl.dd_uniform:.3e} cells/step)",
                       "cells": cells, "parallelism": f"replicas x{world}",
                       "l2": "inputs larger than L2 (c, e, u, v, w: %.2f GB resident)" % (
                           (wl.c.nbytes + wl.e.nbytes + h2d) / 1e9),
                       "algorithmic_bytes_per_cell_step": STEP_BYTES_PER_CELL,
                       "hbm_roofline_frac_step": round(value / world * STEP_BYTES_PER_CELL / peak, 4)},
            "roofline": {"bound": "alu", "kernel": "k_walk (sweep x, y, z)", "achieved": round(fp64_achieved, 4),
                         "peak": round(fp64_peak, 4),
                         "unit": "TFLOP/s",
                         "frac": round(fp64_achieved / fp64_peak, 4),
                         "traffic": traffic,
                         "peak_kind": ("measured: FP64 fused multiply-add chains on every SM (vof_fp64_probe), "
                                       "2 flop each" if fp64 else
                                       "derived: 152 SMs x 2 FP64 FMA per clock x 2 flop x max SM clock"),
                         "fp64_probe": fp64,
                         "peak_derived_tflops": round(fp64_peak_tflops(clocks["sm_max_mhz"] if clocks else None), 4),
                         "flop_per_face": FACE_FLOP, "faces_per_launch": round(faces_per_step / 3),
                         "fp64_issue_frac": round(fp64_achieved / fp64_peak * 2 * FACE_INSTR / FACE_FLOP, 4),
                         "ms_per_launch": round(faces_ms / 3, 5),
                         "share_of_step": round(faces_ms / step_ms_prof, 4) if step_ms_prof > 0 else None,
                         "hbm_frac_step": round(value / world * STEP_BYTES_PER_CELL / peak, 4), "hbm_peak_gbs": peak,
                         "hbm_frac_step_nominal": round(value / world * STEP_BYTES_PER_CELL / HBM_NOMINAL_GBS, 4),
                         "hbm_nominal_gbs": HBM_NOMINAL_GBS},
            "work_counts": counts,
            "kernel_ms": {k: round(v_, 5) for k, v_ in sorted(kern_ms.items(), key=lambda kv: -kv[1])},
            "e2e": {"value": round(e2e_value, 4), "unit": UNIT, "h2d_bytes_per_step": h2d,
                    "d2h_bytes_per_step": P.VOF_NSUMS * 8},
            "gpu_launches": kernels_per_step * args.steps,
            "clocks": clocks,
            "cpu_baseline": cpu,
            "precision_form": pform,
            "learned_form": learned,
            "batched_form": batched,
            "mass_transfer": mt,
            "scheme_le": le,
            "final_sums": [float(x) for x in sums],
        }
        print(json.dumps(out), flush=True)
    if world > 1:
        dist.destroy_process_group()


# conductivities of water and steam at 1 atm (W/m/K) and the latent heat of
# the bubble workload: the scale of mdot only
K_L_WATER, K_G_STEAM = 0.68, 0.025
# droplet boxes of the grouped step that --kernels-once runs (a few GB)
KERNELS_ONCE_BOXES = 64


def mass_transfer_measure(P, g, wl, c, e, stream, barrier, reps=20):
    """vof_mass_transfer on the initial state of the step's workload: the
    mean time of one call over `reps` calls (CUDA events on the launching
    stream), its kernels' shares, and its work counts.  Writes mdot and the
    Step-2 shift dd = -mdot dt / (rho_l h)."""
    import torch
    from paper_2001_03477_gb300 import workloads as W
    ws = torch.empty(P.vof_mass_transfer_workspace_bytes(g), dtype=torch.uint8, device=c.device)
    mdot = torch.empty_like(c)
    dd = torch.empty_like(c)
    dd_per_mdot = -wl.dt / (W.RHO_L * wl.h)
    for _ in range(3):
        P.vof_mass_transfer(g, c, e, K_L_WATER, K_G_STEAM, W.H_FG_WATER, mdot, None, None, dd_per_mdot, dd,
                            workspace=ws, stream=stream)
    barrier()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    for _ in range(reps):
        P.vof_mass_transfer(g, c, e, K_L_WATER, K_G_STEAM, W.H_FG_WATER, mdot, None, None, dd_per_mdot, dd,
                            workspace=ws, stream=stream)
    ev1.record(stream)
    barrier()
    ms = ev0.elapsed_time(ev1) / reps
    P.vof_profile_begin(stream)
    for _ in range(reps):
        P.vof_mass_transfer(g, c, e, K_L_WATER, K_G_STEAM, W.H_FG_WATER, mdot, None, None, dd_per_mdot, dd,
                            workspace=ws, stream=stream)
    launches = P.vof_profile_end()
    kms = {}
    for name, t in launches:
        kms[name] = kms.get(name, 0.0) + t / reps
    counts = P.vof_mass_transfer_work_counts(g, ws, stream)
    # the velocity extension driven by this mdot (Sec. 3.3.1; its CG loop
    # reads the residual on the host, so it is timed on the host clock)
    nz, ny, nx = c.shape
    xw = torch.empty(P.vof_velocity_extension_workspace_bytes(g), dtype=torch.uint8, device=c.device)
    ut = torch.empty((nz, ny, nx + 1), dtype=torch.float64, device=c.device)
    vt = torch.empty((nz, ny + 1, nx), dtype=torch.float64, device=c.device)
    wt = torch.empty((nz + 1, ny, nx), dtype=torch.float64, device=c.device)
    P.vof_velocity_extension(g, c, mdot, W.RHO_L, W.RHO_G, wl.dt, ut=ut, vt=vt, wt=wt, workspace=xw, stream=stream)
    barrier()
    t0 = time.perf_counter()
    ext_reps = 5
    for _ in range(ext_reps):
        ext_it, ext_res = P.vof_velocity_extension(g, c, mdot, W.RHO_L, W.RHO_G, wl.dt, ut=ut, vt=vt, wt=wt,
                                                   workspace=xw, stream=stream)
    barrier()
    ext_ms = (time.perf_counter() - t0) * 1e3 / ext_reps
    # the implicit interface-Dirichlet heat diffusion of the same state
    # (Sec. 3.4.2), host-timed (its Jacobi loop reads the largest change on
    # the host); a failure here is reported in the line, not raised
    try:
        dw = torch.empty(P.vof_heat_diffusion_workspace_bytes(g), dtype=torch.uint8, device=c.device)
        e_d = e.clone()
        P.vof_heat_diffusion(g, c, e_d, K_L_WATER, K_G_STEAM, wl.dt, tol=1e-9, max_iter=1000, workspace=dw,
                             stream=stream)
        barrier()
        t0 = time.perf_counter()
        dif_reps = 3
        for _ in range(dif_reps):
            e_d.copy_(e)
            dif_it, dif_ch = P.vof_heat_diffusion(g, c, e_d, K_L_WATER, K_G_STEAM, wl.dt, tol=1e-9,
                                                  max_iter=1000, workspace=dw, stream=stream)
        barrier()
        dif = {"ms_per_call": round((time.perf_counter() - t0) * 1e3 / dif_reps, 4), "jacobi_sweeps": dif_it,
               "last_change_K": dif_ch,
               "max_abs_dT_K": float(((e_d - e) / (g.Cp_l * c + g.Cp_g * (1 - c))).abs().max())}
        del dw, e_d
    except Exception as exc:  # noqa: BLE001 -- reported, the step's figures stand
        dif = {"error": str(exc)[:200]}
    mixed = (c > g.eps_mixed) & (c < 1 - g.eps_mixed)
    md = mdot[mixed]
    cells = c.numel()
    return {"workload": "the step's workload, initial state (water k_l = 0.68, steam k_g = 0.025 W/m/K)",
            "value": round(cells / (ms * 1e-3) / 1e9, 4), "unit": UNIT, "ms_per_call": round(ms, 5),
            "work_counts": counts, "kernel_ms": {k: round(v_, 5) for k, v_ in kms.items()},
            "launches_per_call": len(launches) // reps,
            "mdot_range": [float(md.min()), float(md.max())] if md.numel() else None,
            "dd_range": [float(dd[mixed].min()), float(dd[mixed].max())] if md.numel() else None,
            "velocity_extension": {"ms_per_call": round(ext_ms, 4), "cg_iterations": ext_it,
                                   "residual": ext_res, "max_abs_correction": float(wt.abs().max())},
            "heat_diffusion": dif}


def scheme_le_measure(P, wl, c0, e0, u, v, w, stream, barrier, steps=100):
    """vof_step with vof_grid.scheme = VOF_SCHEME_LE on the same workload
    and initial state: Gcell/s over `steps` in-place steps (CUDA events)
    after 3 warm-up steps."""
    import torch
    g = P.Grid(wl.shape[2], wl.shape[1], wl.shape[0], wl.bc, wl.h, wl.Cp_l, wl.Cp_g, wl.T_sat,
               scheme=P.VOF_SCHEME_LE)
    st = P.Stepper(g, device=c0.device)
    c, e = c0.clone(), e0.clone()
    for s in range(3):
        st.step(c, e, u, v, w, wl.dt, s, dd_uniform=wl.dd_uniform)
    barrier()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    for s in range(steps):
        st.step(c, e, u, v, w, wl.dt, 3 + s, dd_uniform=wl.dd_uniform)
    ev1.record(stream)
    barrier()
    ms = ev0.elapsed_time(ev1) / steps
    return {"workload": "the step's workload and initial state, Lagrangian-explicit sweeps (Li / CIAM)",
            "steps": steps, "value": round(c.numel() / (ms * 1e-3) / 1e9, 4), "unit": UNIT,
            "ms_per_step": round(ms, 5)}


def fp64_rate(P, dev, stream, iters=20000, blocks=152 * 8):
    """Measured FP64 rate of the part: the library's FP64 probe (8
    independent chains of fused multiply-adds, or adds, per thread on every
    SM), best of 3 launches timed with CUDA events on the launching stream."""
    import torch
    out = torch.empty(blocks * 256, dtype=torch.float64, device=dev)
    res = {}
    for op, name, flop in ((0, "dfma", 2), (1, "dadd", 1)):
        P.vof_fp64_probe(op, 1000, blocks, out, stream)
        best = None
        for _ in range(3):
            ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            ev0.record(stream)
            P.vof_fp64_probe(op, iters, blocks, out, stream)
            ev1.record(stream)
            ev1.synchronize()
            ms = ev0.elapsed_time(ev1)
            best = ms if best is None else min(best, ms)
        ops = blocks * 256 * 8 * iters
        res[name + "_tflops"] = round(ops * flop / (best * 1e-3) / 1e12, 4)
        res[name + "_ginstr_per_s"] = round(ops / (best * 1e-3) / 1e9, 2)
    return res


def dense_roofline(P, st, g, c, e, u, v, w, dt, stream, fp64_peak, hbm_peak, value, reps=3):
    """The FP64 step's kernels on a workload where T varies everywhere (no
    quiet tiles): per-launch times of `reps` steps (CUDA events recorded by
    the library after each launch), faces evaluated, and k_walk's FP64 rate
    against the measured peak; the step against the HBM ledger."""
    import torch
    torch.cuda.synchronize()
    P.vof_profile_begin(stream)
    for r in range(reps):
        st.step(c, e, u, v, w, dt, r)
    launches = P.vof_profile_end()
    kms = {}
    for name, t in launches:
        kms[name] = kms.get(name, 0.0) + t / reps
    counts = P.vof_step_work_counts(g, st.workspace, stream)
    faces_ms = sum(kms.get(f"sweep_{a}.walk", 0.0) for a in "xyz")
    faces = sum(counts["faces"])
    ach = FACE_FLOP * faces / (faces_ms * 1e-3) / 1e12 if faces_ms > 0 else 0.0
    return {"kernel": "k_walk (sweep x, y, z)", "bound": "alu", "unit": "TFLOP/s", "achieved": round(ach, 4),
            "peak": round(fp64_peak, 4), "frac": round(ach / fp64_peak, 4), "flop_per_face": FACE_FLOP,
            "fp64_issue_frac": round(ach / fp64_peak * 2 * FACE_INSTR / FACE_FLOP, 4),
            "faces_per_launch": round(faces / 3), "ms_per_launch": round(faces_ms / 3, 5),
            "share_of_step": round(faces_ms / sum(kms.values()), 4),
            "hbm_frac_step": round(value * STEP_BYTES_PER_CELL / hbm_peak, 4), "work_counts": counts,
            "kernel_ms": {k: round(v_, 5) for k, v_ in sorted(kms.items(), key=lambda kv: -kv[1])}}


def precision_form(dev, steps=20, n=512, fp64_peak=None, hbm_peak=None):
    """The precision form against the FP64 form on the 512^3 deformation
    workload (sphere R = 0.15 in the LeVeque field, smooth random T, no
    phase change): Gcell/s of each (CUDA events around `steps` in-place
    steps from the same initial state) and the difference of the two final
    states, with the totals each form conserves; and the FP64 step's
    kernels on this dense workload (T varies in every cell)."""
    import torch
    import paper_2001_03477_gb300 as P
    from paper_2001_03477_gb300 import workloads as W
    t0 = time.perf_counter()
    wl = W.deformation_sphere(n=n, nsub=8)
    gen_s = time.perf_counter() - t0
    c0 = torch.from_numpy(wl.c).to(dev)
    e0 = torch.from_numpy(wl.e).to(dev)
    u, v, w = (torch.from_numpy(a).to(dev) for a in (wl.u, wl.v, wl.w))
    del wl.c, wl.e, wl.u, wl.v, wl.w
    stream = torch.cuda.current_stream(dev)
    res, finals = {}, {}
    for name, prec in (("f64", P.VOF_F64), ("f32_flux", P.VOF_F32_FLUX)):
        g = P.Grid(n, n, n, wl.bc, wl.h, wl.Cp_l, wl.Cp_g, wl.T_sat, precision=prec)
        st = P.Stepper(g, device=dev)
        c, e = c0.clone(), e0.clone()
        for s in range(3):
            st.step(c, e, u, v, w, wl.dt, s, dd_uniform=0.0)
        c.copy_(c0); e.copy_(e0)
        clip = torch.zeros((), dtype=torch.float64, device=dev)
        torch.cuda.synchronize(dev)
        ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        ev0.record(stream)
        for s in range(steps):
            st.step(c, e, u, v, w, wl.dt, s, dd_uniform=0.0)
        ev1.record(stream)
        torch.cuda.synchronize(dev)
        ms = ev0.elapsed_time(ev1)
        # the same steps again from the initial state, adding up the clipped
        # volume of every step (outside the timed region)
        c.copy_(c0); e.copy_(e0)
        for s in range(steps):
            st.step(c, e, u, v, w, wl.dt, s, dd_uniform=0.0)
            clip += st.sums[2]
        sums = st.sums.cpu().numpy()
        res[name] = {"value": round(n ** 3 * steps / (ms * 1e-3) / 1e9, 4), "ms_per_step": round(ms / steps, 5),
                     "sum_c": float(sums[0]), "sum_e": float(sums[1]), "clipped": float(clip)}
        if name == "f64" and fp64_peak:
            cx, ex = c0.clone(), e0.clone()
            dense = dense_roofline(P, st, g, cx, ex, u, v, w, wl.dt, stream, fp64_peak, hbm_peak,
                                   res[name]["value"])
            del cx, ex
        finals[name] = (c, e)
        del st
    sc0 = float(c0.sum())
    se0 = float(e0.sum())
    cd, ed = finals["f64"]
    cf, ef = finals["f32_flux"]
    dc = (cf - cd).abs()
    Tmax = float((ed / (wl.Cp_l * cd + wl.Cp_g * (1 - cd))).max())
    out = {
        "workload": f"deformation-sphere {n}^3 (R=0.15 at (0.35,0.35,0.35), LeVeque field t=0, CFL 0.5, "
                    f"water/steam Cp ratio {wl.Cp_l / wl.Cp_g:.1f}, T = 1 + 8 seeded Fourier modes, no shift)",
        "steps": steps, "unit": UNIT,
        "value": res["f32_flux"]["value"], "value_fp64": res["f64"]["value"],
        "speedup": round(res["f32_flux"]["value"] / res["f64"]["value"], 4),
        "vs_fp64": {
            "max_abs_dc": float(dc.max()),
            "cells_abs_dc_gt_1e-6": int((dc > 1e-6).sum()),
            "interface_cells": int(((cd > 0) & (cd < 1)).sum()),
            "max_abs_de_over_Cpl_Tmax": float((ef - ed).abs().max()) / (wl.Cp_l * Tmax),
            "sum_c_rel_diff": (res["f32_flux"]["sum_c"] - res["f64"]["sum_c"]) / res["f64"]["sum_c"],
            "sum_e_rel_diff": (res["f32_flux"]["sum_e"] - res["f64"]["sum_e"]) / res["f64"]["sum_e"],
        },
        # volume changes only by the clipped volume (no shift, divergence-free
        # face velocities, none through the boundary): drift = what is left
        "mass_drift_rel": {k: (r["sum_c"] - sc0 - r["clipped"]) / sc0 for k, r in res.items()},
        "energy_drift_rel": {k: (r["sum_e"] - se0) / se0 for k, r in res.items()},
        "input_generation_s": round(gen_s, 1),
    }
    if fp64_peak:
        out["roofline_fp64_dense"] = dense
    return out


def _training_part(n, seed, start):
    from paper_2001_03477_gb300 import workloads as W
    return W.training_stencils(n, seed=seed, start=start)


def training_set(count, seed=50):
    """`count` training stencils of the learned normal (spheres, ellipsoids,
    planes; workloads.training_stencils) generated on all host cores by a
    spawn pool (each range of sample indices from its own seeded streams)."""
    import multiprocessing as mp
    nproc = os.cpu_count() or 1
    chunk = max(2048, -(-count // (nproc * 4)))
    jobs = [(min(chunk, count - s), seed, s) for s in range(0, count, chunk)]
    with mp.get_context("spawn").Pool(nproc) as pool:
        parts = pool.starmap(_training_part, jobs)
    return np.concatenate([p[0] for p in parts]), np.concatenate([p[1] for p in parts]), nproc


def _angles_deg(m, y):
    m = np.asarray(m, dtype=np.float64)
    cosv = np.sum(m * y, axis=1) / (np.linalg.norm(m, axis=1) * np.linalg.norm(y, axis=1))
    return np.degrees(np.arccos(np.clip(cosv, -1.0, 1.0)))


def shape_error_run(P, g, c0, e0, u0, v0, w0, dt, nsteps, dev, period=3.0):
    """L1 shape error sum |c(T) - c(0)| h^3 after one full period of the
    LeVeque field (the velocity of step s is the t = 0 field times
    cos(pi t / T) at t = (s + 1/2) dt), and the step rate."""
    import torch
    st = P.Stepper(g, device=dev)
    c, e = c0.clone(), e0.clone()
    u, v, w = torch.empty_like(u0), torch.empty_like(v0), torch.empty_like(w0)
    stream = torch.cuda.current_stream(dev)
    torch.cuda.synchronize(dev)
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    for s in range(nsteps):
        gt = math.cos(math.pi * (s + 0.5) * dt / period)
        torch.mul(u0, gt, out=u)
        torch.mul(v0, gt, out=v)
        torch.mul(w0, gt, out=w)
        st.step(c, e, u, v, w, dt, s)
    ev1.record(stream)
    torch.cuda.synchronize(dev)
    counts = P.vof_step_work_counts(g, st.workspace, stream)
    err = float((c - c0).abs().sum()) * g.h ** 3
    return {"l1_shape_error": err, "rel_to_volume": err / (float(c0.sum()) * g.h ** 3),
            "ms_per_step": round(ev0.elapsed_time(ev1) / nsteps, 5), "last_step_mlp_fallback": counts["mlp_fallback"],
            "last_step_mixed": counts["mixed"]}


def learned_form(dev, fp64_peak=None, n=512, steps=20, ntrain=1_000_000, train_steps=8000, batch=16384,
                 n_shape=128):
    """The learned-normal form (the sweeps' MYC normals replaced by the
    27-64-64-3 network on the tensor cores, MYC as fallback), against the
    plain FP64 form:
      * training on the GPU (the library's forward, backward and Adam
        kernels) on `ntrain` generated stencils, and the trained network's
        mean angular error on held-out sphere stencils against MYC's;
      * throughput at n^3 on the deformation sphere with the phase-change
        shift dd = -0.01 (precision form + learned normals vs FP64 + MYC)
        and the volume drift over `steps` steps;
      * the L1 shape error after a full period of the LeVeque field at
        n_shape^3 for the learned, MYC and Youngs normals."""
    import torch
    import paper_2001_03477_gb300 as P
    from paper_2001_03477_gb300 import workloads as W
    t0 = time.perf_counter()
    X, Y, nproc = training_set(ntrain)
    gen_s = time.perf_counter() - t0
    Xd, Yd = torch.from_numpy(X).to(dev), torch.from_numpy(Y).to(dev)
    del X, Y
    mlp = P.MLP(P.MLP.init_master(5), device=dev)
    loss = torch.zeros(1, dtype=torch.float32, device=dev)
    stream = torch.cuda.current_stream(dev)
    hist = []
    torch.cuda.synchronize(dev)
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    for s in range(train_steps):
        lr = 3e-3 if s < train_steps // 2 else (1e-3 if s < (4 * train_steps) // 5 else 3e-4)
        mlp.train_step(Xd, Yd, batch, lr, seed=50, loss=loss)
        if s % (train_steps // 16) == 0 or s == train_steps - 1:
            hist.append((s, loss.clone()))
    ev1.record(stream)
    torch.cuda.synchronize(dev)
    train_ms = ev0.elapsed_time(ev1)
    hist = [(s, float(l_.item())) for s, l_ in hist]
    del Xd, Yd
    # held-out sphere stencils: learned (with fallback) against MYC alone
    # (a zero network has no usable normal, so it falls back everywhere)
    Xt, Yt = W.training_stencils(3000, seed=99, kinds=("sphere",))
    Xtd = torch.from_numpy(Xt).to(dev)
    zero = P.MLP(np.zeros(P.VOF_MLP_PARAMS, dtype=np.float32), device=dev)
    out = {}
    for name, net in (("learned", mlp), ("myc", zero)):
        m = torch.zeros((len(Xt), 3), dtype=torch.float64, device=dev)
        fb = torch.zeros(len(Xt), dtype=torch.uint8, device=dev)
        P.vof_mlp_normals(net.packed, Xtd, m, fb)
        ang = _angles_deg(m.cpu().numpy(), Yt)
        out[name] = {"mean_deg": round(float(ang.mean()), 4), "median_deg": round(float(np.median(ang)), 4),
                     "p99_deg": round(float(np.percentile(ang, 99)), 4), "fallback_frac": float(fb.float().mean())}
    training = {"stencils": ntrain, "generation_s": round(gen_s, 1), "generation_procs": nproc,
                "steps": train_steps, "batch": batch, "samples_per_s": round(train_steps * batch / (train_ms * 1e-3)),
                "ms_per_step": round(train_ms / train_steps, 4), "loss": hist,
                "held_out_spheres": out}
    # ---- throughput on the deformation sphere with the shift -------------
    wl = W.deformation_sphere(n=n, nsub=8)
    c0 = torch.from_numpy(wl.c).to(dev)
    e0 = torch.from_numpy(wl.e).to(dev)
    u, v, w = (torch.from_numpy(a).to(dev) for a in (wl.u, wl.v, wl.w))
    del wl.c, wl.e, wl.u, wl.v, wl.w
    dd = -0.01
    forms = {"fp64_myc": dict(precision=P.VOF_F64, normal=P.VOF_NORMAL_MYC),
             "f32_learned": dict(precision=P.VOF_F32_FLUX, normal=P.VOF_NORMAL_MLP, mlp=mlp.packed)}
    res = {}
    sc0 = float(c0.sum())
    for name, kw in forms.items():
        g = P.Grid(n, n, n, wl.bc, wl.h, wl.Cp_l, wl.Cp_g, wl.T_sat, **kw)
        st = P.Stepper(g, device=dev)
        c, e = c0.clone(), e0.clone()
        for s in range(3):
            st.step(c, e, u, v, w, wl.dt, s, dd_uniform=dd)
        c.copy_(c0); e.copy_(e0)
        torch.cuda.synchronize(dev)
        ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        ev0.record(stream)
        for s in range(steps):
            st.step(c, e, u, v, w, wl.dt, s, dd_uniform=dd)
        ev1.record(stream)
        torch.cuda.synchronize(dev)
        ms = ev0.elapsed_time(ev1)
        # volume bookkeeping of the same steps: sum c changes only by the
        # clipped volume and the shift's sum dc (closed box)
        c.copy_(c0); e.copy_(e0)
        book = 0.0
        for s in range(steps):
            sums = st.step(c, e, u, v, w, wl.dt, s, dd_uniform=dd).cpu().numpy()
            book += -sums[2] + sums[3]
        counts = P.vof_step_work_counts(g, st.workspace, stream)
        res[name] = {"value": round(n ** 3 * steps / (ms * 1e-3) / 1e9, 4), "ms_per_step": round(ms / steps, 5),
                     "mass_drift_rel": (float(sums[0]) - sc0 - book) / sc0,
                     "mlp_fallback_last_step": counts["mlp_fallback"], "mixed_last_step": counts["mixed"]}
        del st, c, e
    del c0, e0, u, v, w
    torch.cuda.empty_cache()
    # ---- shape error after a full period at n_shape^3 ---------------------
    ws = W.deformation_sphere(n=n_shape, nsub=8)
    dts = 0.25 * ws.h / 2.0  # face CFL 0.25 (max |u| = 2)
    nper = int(round(3.0 / dts))
    cs = torch.from_numpy(ws.c).to(dev)
    es = torch.from_numpy((ws.Cp_l * ws.c + ws.Cp_g * (1 - ws.c)) * 1.0).to(dev)  # uniform T: c alone matters
    us, vs, wsf = (torch.from_numpy(a).to(dev) for a in (ws.u, ws.v, ws.w))
    shape = {}
    for name, kw in (("learned_f32", dict(precision=P.VOF_F32_FLUX, normal=P.VOF_NORMAL_MLP, mlp=mlp.packed)),
                     ("myc_f64", dict(precision=P.VOF_F64, normal=P.VOF_NORMAL_MYC)),
                     ("myc_f32", dict(precision=P.VOF_F32_FLUX, normal=P.VOF_NORMAL_MYC)),
                     ("youngs_f64", dict(precision=P.VOF_F64, normal=P.VOF_NORMAL_YOUNGS))):
        g = P.Grid(n_shape, n_shape, n_shape, ws.bc, ws.h, ws.Cp_l, ws.Cp_g, ws.T_sat, **kw)
        shape[name] = shape_error_run(P, g, cs, es, us, vs, wsf, dts, nper, dev)
    return {"workload": f"deformation-sphere {n}^3 (R=0.15 at (0.35,0.35,0.35), LeVeque field t=0, CFL 0.5, "
                        f"water/steam Cp ratio {wl.Cp_l / wl.Cp_g:.1f}, T = 1 + 8 seeded Fourier modes) with the "
                        f"phase-change shift dd = {dd} in every mixed cell",
            "steps": steps, "unit": UNIT,
            "value": res["f32_learned"]["value"], "value_fp64_myc": res["fp64_myc"]["value"],
            "speedup_vs_fp64": round(res["f32_learned"]["value"] / res["fp64_myc"]["value"], 4),
            "forms": res, "training": training,
            "shape_error_full_period": {"grid": f"{n_shape}^3", "steps": nper, "dt": dts, "forms": shape}}


def _droplet_part(indices, nsub):
    from paper_2001_03477_gb300 import workloads as W
    out = []
    for i in indices:
        wl = W.droplet_subdomain(i, nsub=nsub)
        vel = (float(wl.u.flat[0]), float(wl.v.flat[0]), float(wl.w.flat[0]))
        out.append((wl.c, wl.h, wl.dt, wl.dd_uniform, vel))
    return out


def batched_form(dev, nbox=4096, nsub=4, steps=5):
    """The batched droplet workload: `nbox` independent periodic boxes of
    edge U{24..96} (about 1.2e9 cells for 4096), one sphere or ellipsoid
    each, uniform velocity |u| <= 1 at CFL 0.25, shift dd ~ U(-0.02, 0.02)
    (workloads.droplet_subdomain, volume fractions on nsub^2 chords per
    cell, generated on all host cores).  The grouped form (vof_group_*: one
    launch per kernel of the step over all boxes, the CTA granularity picked
    by the autotuner on a sample) timed directly and as a CUDA-graph replay;
    beside it vof_batched_step over lane streams (12 launches per box).
    CUDA events on the launching stream."""
    import multiprocessing as mp
    import torch
    import paper_2001_03477_gb300 as P
    t0 = time.perf_counter()
    nproc = os.cpu_count() or 1
    chunks = [list(range(s, min(s + 32, nbox))) for s in range(0, nbox, 32)]
    with mp.get_context("spawn").Pool(nproc) as pool:
        parts = pool.starmap(_droplet_part, [(ch, nsub) for ch in chunks])
    gen_s = time.perf_counter() - t0
    boxes = []
    cells = 0
    for part in parts:
        for c, h, dt, dd, vel in part:
            n = c.shape[0]
            cd = torch.from_numpy(c).to(dev)
            g = P.Grid(n, n, n, (0, 0, 0), h, 1000.0, 1.0, 1.0)
            u = torch.full((n, n, n + 1), vel[0], dtype=torch.float64, device=dev)
            v = torch.full((n, n + 1, n), vel[1], dtype=torch.float64, device=dev)
            w = torch.full((n + 1, n, n), vel[2], dtype=torch.float64, device=dev)
            boxes.append(P.Box(g, cd, 1000.0 * cd, u, v, w, dt, None, dd))
            cells += n ** 3
    del parts
    stream = torch.cuda.current_stream(dev)
    # ---- grouped: one launch per kernel of the step over all boxes --------
    t1 = time.perf_counter()
    work, wtimes = P.Group.autotune(boxes[:512], candidates=(1024, 4096, 16384), steps=2, device=dev)
    tune_s = time.perf_counter() - t1
    grp = P.Group(boxes, work, dev)
    for s in range(2):
        grp.step(s)
    torch.cuda.synchronize(dev)
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    for s in range(steps):
        grp.step(2 + s)
    ev1.record(stream)
    torch.cuda.synchronize(dev)
    grp_ms = ev0.elapsed_time(ev1) / steps
    P.vof_profile_begin(stream)
    grp.step(0)
    gl = P.vof_profile_end()
    grp_kernel_ms = {}
    for name, t in gl:
        grp_kernel_ms[name] = round(grp_kernel_ms.get(name, 0.0) + t, 4)
    cap = torch.cuda.Stream(dev)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=cap):
        grp.step(0, stream=cap)
    graph.replay()
    torch.cuda.synchronize(dev)
    ev0.record(stream)
    for s in range(steps):
        graph.replay()
    ev1.record(stream)
    torch.cuda.synchronize(dev)
    grp_graph_ms = ev0.elapsed_time(ev1) / steps
    gsums = grp.sums.cpu().numpy()
    grp_ws_gb = grp.workspace.numel() / 1e9
    grp.close()
    del grp, graph
    torch.cuda.empty_cache()
    # ---- lanes: one vof_step per box on concurrent streams ----------------
    batch = P.BoxBatch(boxes, 8, dev)
    lanes = batch.autotune(candidates=(4, 8, 16, 32), sample=512, steps=2)
    for s in range(2):
        batch.step(s)
    torch.cuda.synchronize(dev)
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    for s in range(steps):
        batch.step(2 + s)
    ev1.record(stream)
    torch.cuda.synchronize(dev)
    direct_ms = ev0.elapsed_time(ev1) / steps
    # one step captured (the lanes become parallel branches of the graph)
    cap = torch.cuda.Stream(dev)
    graph = torch.cuda.CUDAGraph()
    t1 = time.perf_counter()
    with torch.cuda.graph(graph, stream=cap):
        batch.step(0, stream=cap)
    graph.replay()
    torch.cuda.synchronize(dev)
    inst_s = time.perf_counter() - t1
    ev0.record(stream)
    for s in range(steps):
        graph.replay()
    ev1.record(stream)
    torch.cuda.synchronize(dev)
    graph_ms = ev0.elapsed_time(ev1) / steps
    sums = batch.sums.cpu().numpy()
    return {"workload": f"{nbox} periodic droplet boxes, edge U{{24..96}} (one sphere or ellipsoid each, uniform "
                        f"|u| <= 1 at CFL 0.25, dd ~ U(-0.02, 0.02), C_pl:C_pg 1000), {cells} cells",
            "cells": cells, "unit": UNIT,
            "value": round(cells / (grp_ms * 1e-3) / 1e9, 4), "ms_per_step": round(grp_ms, 3),
            "grouped": {"work_per_cta": work, "autotune_s_per_step": {str(k): round(v_, 5) for k, v_ in wtimes.items()},
                        "autotune_s": round(tune_s, 1), "launches_per_step": len(gl),
                        "value_graph_replay": round(cells / (grp_graph_ms * 1e-3) / 1e9, 4),
                        "ms_per_step_graph_replay": round(grp_graph_ms, 3), "kernel_ms": grp_kernel_ms,
                        "workspace_gb": round(grp_ws_gb, 2), "finite": bool(np.isfinite(gsums).all())},
            "lanes": {"lanes": lanes, "autotune_s_per_step": {str(k): round(v_, 5) for k, v_ in batch.timings.items()},
                      "value": round(cells / (direct_ms * 1e-3) / 1e9, 4), "ms_per_step": round(direct_ms, 3),
                      "value_graph_replay": round(cells / (graph_ms * 1e-3) / 1e9, 4),
                      "graph_capture_and_instantiate_s": round(inst_s, 2),
                      "launches_per_step": "12 per box (one vof_step each)",
                      "finite": bool(np.isfinite(sums).all())},
            "input_generation_s": round(gen_s, 1)}


def oracle_sample(nz_slab=8):
    """A bounded sample of the workload for the CPU oracle: the z-slab of
    nz_slab planes through the bubble centre (interface-rich), with its own
    face velocities; returns the oracle grid and arrays."""
    import oracle as O
    wl = load_workload()
    n = N_CELLS
    k0 = n // 2 - nz_slab // 2
    c = np.ascontiguousarray(wl.c[k0:k0 + nz_slab])
    e = np.ascontiguousarray(wl.e[k0:k0 + nz_slab])
    u = np.ascontiguousarray(wl.u[k0:k0 + nz_slab])
    v = np.ascontiguousarray(wl.v[k0:k0 + nz_slab])
    w = np.ascontiguousarray(wl.w[k0:k0 + nz_slab + 1])
    g = O.Grid(n, n, nz_slab, wl.bc, wl.h, wl.Cp_l, wl.Cp_g, wl.T_sat)
    return O, g, wl, c, e, u, v, w


def cpu_model():
    """The host CPU's model name (lscpu, else /proc/cpuinfo), or None."""
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.strip().startswith("Model name"):
                return line.split(":", 1)[1].strip()
    except Exception:  # noqa: BLE001 -- informative only
        pass
    try:
        with open("/proc/cpuinfo") as f:
            for line in f:
                if line.lower().startswith(("model name", "cpu part")):
                    return line.split(":", 1)[1].strip()
    except OSError:
        pass
    return None


def _oracle_rate(O, g, wl, c, e, u, v, w, budget_s):
    t0 = time.perf_counter()
    steps = 0
    while True:
        c, e, _ = O.step(g, c, e, u, v, w, wl.dt, steps, dd_uniform=wl.dd_uniform)
        steps += 1
        if time.perf_counter() - t0 > budget_s:
            break
    dt = time.perf_counter() - t0
    return c.size * steps / dt / 1e9, steps, dt


def cpu_baseline(budget_s=12.0):
    """The oracle (as it stands) on the host cores: all cores (OpenMP over
    the per-cell loops; bit-identical to one thread) and one thread, on the
    256 x 256 x 8 z-slab through the bubble centre."""
    O, g, wl, c, e, u, v, w = oracle_sample()
    nproc = os.cpu_count() or 1
    O.set_threads(nproc)
    v_all, s_all, t_all = _oracle_rate(O, g, wl, c, e, u, v, w, budget_s)
    O.set_threads(1)
    v_one, s_one, t_one = _oracle_rate(O, g, wl, c, e, u, v, w, budget_s)
    O.set_threads(nproc)
    cells = c.size
    return {"value": round(v_all, 6), "unit": UNIT, "cores": nproc, "kind": "oracle",
            "sample": f"{s_all} oracle steps on the 256x256x8 z-slab through the bubble centre "
                      f"({cells} cells, {t_all:.1f} s, {nproc} threads)",
            "cpu_model": cpu_model(), "nproc": nproc,
            "single_thread": {"value": round(v_one, 6), "unit": UNIT, "cores": 1,
                              "sample": f"{s_one} steps of the same slab, {t_one:.1f} s"}}


def run_reference(args):
    rank, world, local = dist_env()
    if rank != 0:
        return
    O, g, wl, c, e, u, v, w = oracle_sample(nz_slab=2)
    O.set_threads(1)
    for s in range(args.warmup):
        c, e, _ = O.step(g, c, e, u, v, w, wl.dt, s, dd_uniform=wl.dd_uniform)
    t0 = time.perf_counter()
    for s in range(args.steps):
        c, e, _ = O.step(g, c, e, u, v, w, wl.dt, args.warmup + s, dd_uniform=wl.dd_uniform)
    dt = time.perf_counter() - t0
    cells = c.size
    value = cells * args.steps / dt / 1e9
    sample = (f"each step: one oracle step on the 256x256x2 z-slab through the bubble centre ({cells} cells), "
              f"single thread")
    out = {"impl": "reference", "metric": METRIC, "value": round(value, 6), "unit": UNIT, "n_gpus": world,
           "steps": args.steps, "warmup": args.warmup, "ms_per_step": dt * 1e3 / args.steps,
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
           "config": {"workload": f"bubble-growth {N_CELLS}^3 (oracle sample)", "cells": cells,
                      "parallelism": "host, 1 thread"},
           "cpu_baseline": {"value": round(value, 6), "unit": UNIT, "cores": 1, "kind": "oracle", "sample": sample},
           "e2e": {"value": round(value, 6), "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(out), flush=True)


def kernels_once():
    """One time step (vof_step, the benchmark's launch configuration) and
    one vof_mass_transfer call on the benchmark workload: the target of the
    committed ncu captures."""
    import torch
    import paper_2001_03477_gb300 as P
    from paper_2001_03477_gb300 import build
    from paper_2001_03477_gb300 import workloads as W
    build.build()
    wl = load_workload()
    g = P.Grid(wl.shape[2], wl.shape[1], wl.shape[0], wl.bc, wl.h, wl.Cp_l, wl.Cp_g, wl.T_sat)
    dev = torch.device("cuda", 0)
    c = torch.from_numpy(wl.c).to(dev)
    e = torch.from_numpy(wl.e).to(dev)
    u, v, w = (torch.from_numpy(a).to(dev) for a in (wl.u, wl.v, wl.w))
    st = P.Stepper(g, device=dev)
    st.step(c, e, u, v, w, wl.dt, 0, dd_uniform=wl.dd_uniform)
    # and one evaluation of the mass transfer rate of the state reached
    mdot = torch.empty_like(c)
    P.vof_mass_transfer(g, c, e, K_L_WATER, K_G_STEAM, W.H_FG_WATER, mdot)
    # the learned normal: one forward pass over 131072 stencils, their
    # normals with the MYC fallback, and one training step of 16384 samples
    rng = np.random.default_rng(0)
    X = torch.from_numpy(rng.random((131072, 27))).to(dev)
    N = torch.nn.functional.normalize(torch.from_numpy(rng.normal(size=(131072, 3))), dim=1).to(dev)
    mlp = P.MLP(P.MLP.init_master(5), device=dev)
    y = torch.empty((131072, 3), dtype=torch.float32, device=dev)
    P.vof_mlp_forward(mlp.packed, X, y)
    m = torch.empty((131072, 3), dtype=torch.float64, device=dev)
    P.vof_mlp_normals(mlp.packed, X, m)
    mlp.train_step(X, N, 16384, 1e-3, seed=1)
    # the two solvers of the state reached: the velocity extension driven by
    # that mdot and the implicit interface-Dirichlet heat diffusion
    nz, ny, nx = c.shape
    ut = torch.empty((nz, ny, nx + 1), dtype=torch.float64, device=dev)
    vt = torch.empty((nz, ny + 1, nx), dtype=torch.float64, device=dev)
    wt = torch.empty((nz + 1, ny, nx), dtype=torch.float64, device=dev)
    ext_it, _ = P.vof_velocity_extension(g, c, mdot, W.RHO_L, W.RHO_G, wl.dt, ut=ut, vt=vt, wt=wt)
    dif_it, _ = P.vof_heat_diffusion(g, c, e.clone(), K_L_WATER, K_G_STEAM, wl.dt, tol=1e-9, max_iter=1000)
    del ut, vt, wt
    # one grouped step of a small droplet batch (the batched form's kernels)
    boxes = []
    for cb, h, dt, dd, vel in _droplet_part(range(KERNELS_ONCE_BOXES), 4):
        n = cb.shape[0]
        cd = torch.from_numpy(cb).to(dev)
        gb = P.Grid(n, n, n, (0, 0, 0), h, 1000.0, 1.0, 1.0)
        boxes.append(P.Box(gb, cd, 1000.0 * cd, torch.full((n, n, n + 1), vel[0], dtype=torch.float64, device=dev),
                           torch.full((n, n + 1, n), vel[1], dtype=torch.float64, device=dev),
                           torch.full((n + 1, n, n), vel[2], dtype=torch.float64, device=dev), dt, None, dd))
    grp = P.Group(boxes, 1024, dev)
    grp.step(0)
    torch.cuda.synchronize()
    gs = grp.sums.cpu().numpy()
    grp.close()
    print("kernels-once ok", [float(x) for x in st.sums.cpu()], float(mdot.sum()), float(y.abs().sum()),
          "extension", ext_it, "diffusion", dif_it, "group", len(boxes), bool(np.isfinite(gs).all()))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=500)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["gpu", "reference"], default="gpu")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-precision-form", action="store_true",
                    help="skip the precision-form comparison on the 512^3 deformation workload")
    ap.add_argument("--no-batched-form", action="store_true",
                    help="skip the batched droplet workload (4096 boxes, ~1.2e9 cells)")
    ap.add_argument("--no-learned-form", action="store_true",
                    help="skip the learned-normal form (GPU training, 512^3 step, full-period shape errors)")
    ap.add_argument("--step-only", action="store_true",
                    help="time the step alone: no precision-form, mass-transfer or Lagrangian-explicit lines "
                         "(the launch list of the step)")
    ap.add_argument("--kernels-once", action="store_true",
                    help="launch each hot-path kernel once on the workload (profiling target)")
    args = ap.parse_args()
    if args.kernels_once:
        kernels_once()
        return
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        run_reference(args)
    else:
        run_gpu(args)


if __name__ == "__main__":
    main()
