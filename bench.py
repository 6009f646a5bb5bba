#!/usr/bin/env python3
"""Throughput of recursive Priori L+S reconstruction (arXiv:1411.6206) on one GB300.

A step is one pass of the whole hot path over one batch of input: the 20-frame cardiac-shaped
sequence (128 x 128 x 16 voxels, 8 coils, 8x variable-density ky-kz undersampling, frame 1
at 50%, 50 iterations of Algorithm 1 per frame, support and singular values passed from frame
to frame). Inputs (coil maps, k-space samples of every frame) are resident in HBM before the
timed region; the per-frame masks are host arrays (the line table is built on the host).

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Prints one JSON line. `value` is whole-job frames/s; under torchrun every rank reconstructs
its own sequence (independent sessions, weak scaling, no data-path collective) and the time
is the maximum over ranks. `--impl reference` times the FP64 CPU oracle on the same workload.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import math
import os
import re
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "recon frames/s and p50/p99 frame latency, served vs plain, at NRMSE≤1e-3"
SM_COUNT = 152
FP32_LANES_PER_SM = 128


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--frames", type=int, default=None, help="frames per step (default: all 20)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--cpu-frames", type=int, default=2, help="oracle frames in the CPU baseline")
    ap.add_argument("--profile", type=int, default=1,
                    help="after the timed steps, one pass with CUDA events around every kernel (roofline)")
    ap.add_argument("--workload", default="cardiac", choices=["cardiac", "precision", "mix160"],
                    help="cardiac: 128x128x16 x 20 frames, 8 coils (default); precision: 192x192x32 x 25, 12 coils; "
                         "mix160: the 160x160x14 x 20, 16-coil member of the serving mix (autotuned runtime kernel)")
    ap.add_argument("--precision", default="fp32", choices=["fp32", "tf32", "bf16"],
                    help="Gram and reprojection arithmetic (tf32/bf16: tensor cores with one refinement step)")
    ap.add_argument("--eig", default=None, choices=["fp32", "fp64"],
                    help="eigendecomposition precision (default fp32 with --precision fp32, else fp64)")
    ap.add_argument("--no-served", action="store_true", help="skip the serving study")
    ap.add_argument("--no-batched", action="store_true", help="skip the batched study")
    ap.add_argument("--serve-seconds", type=float, default=6.5, help="arrival window of the serving study")
    ap.add_argument("--serve-sessions", type=int, default=16)
    ap.add_argument("--batch-problems", type=int, default=64)
    ap.add_argument("--no-sweep", action="store_true", help="skip the serving sweep of arrival rates")
    ap.add_argument("--no-precision", action="store_true", help="skip the precision study (192x192x32, 12 coils)")
    ap.add_argument("--no-small", action="store_true", help="skip the 32x32x8 single-coil latency study")
    ap.add_argument("--precision-frames", type=int, default=5, help="frames per mode in the precision study")
    ap.add_argument("--no-fig3", action="store_true", help="skip the PSNR-vs-sampling study (plain vs Priori L+S)")
    return ap.parse_args()


def peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(p) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), float(d.get("sm_max_mhz", 2070.0)), "measured"
    except Exception:
        return 6800.0, 2070.0, "fallback"


class Clocks:
    """nvidia-smi sampling of SM clock and throttle reasons during the timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.path = None

    def start(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.Q}", "--format=csv,noheader,nounits",
                 "-lms", "100"], stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        rows = []
        with open(self.path) as f:
            for line in f:
                parts = [p.strip() for p in line.split(",")]
                if len(parts) >= 9 and parts[1].replace(".", "").isdigit():
                    rows.append(parts)
        os.unlink(self.path)
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        sm = [float(r[1]) for r in rows]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if r[5 + i].lower() == "active"})
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(float(r[2]) for r in rows),
                "reasons": reasons, "samples": len(rows)}


def source_digest(path):
    """sha256 of a kernel's source and of every file that it includes by name in quotes, and these in
    turn (the transforms of a kernel are in headers of their own), each once, in order of their paths."""
    seen, todo = {}, [os.path.normpath(path)]
    while todo:
        p = todo.pop()
        if p in seen:
            continue
        with open(os.path.join(ROOT, p), "rb") as f:
            seen[p] = f.read()
        for name in re.findall(rb'^\s*#include "([^"]+)"', seen[p], re.M):
            for d in (os.path.dirname(p), "include"):
                q = os.path.normpath(os.path.join(d, name.decode()))
                if os.path.exists(os.path.join(ROOT, q)):
                    todo.append(q)
                    break
    h = hashlib.sha256()
    for p in sorted(seen):
        h.update(p.encode() + b"\0" + seen[p] + b"\0")
    return h.hexdigest()


def profiled_traffic(summary):
    """DRAM bytes per launch from a committed ncu summary under profiles/, or None when the
    kernel's source, or a header of it, has changed since the counters were taken."""
    try:
        kv = {}
        with open(os.path.join(ROOT, "profiles", summary)) as f:
            for line in f:
                if ":" in line and not line[0].isspace():
                    k, v = line.split(":", 1)
                    kv[k.strip()] = v.strip()
        if source_digest(kv["kernel_source"]) != kv["source_sha256"]:
            return None
        return int(kv["dram_bytes_per_launch"])
    except (OSError, KeyError, ValueError):
        return None


def eig_flops_per_launch(n, sweeps=2):
    """Nominal real flops of one eigen/SVT launch for an n x n Gram: per Jacobi sweep (np-1
    steps) every 2 x 2 block is rotated on both sides (16 complex multiply-adds per block) and
    every row pair of V once (8); plus V^H G V for the warm start and W = V f V^H (8 n^3 each)."""
    np_ = n + (n & 1)
    nh = np_ // 2
    step = nh * nh * 16 * 8 + nh * nh * 8 * 8
    return sweeps * (np_ - 1) * step + 3 * 8 * n ** 3


def dist():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


# ------------------------------------------------------------------------------------
# workload
# ------------------------------------------------------------------------------------

def plan_kw(args):
    from paper_1411_6206_gb300 import lps
    prec = {"fp32": lps.FP32, "tf32": lps.TF32_REFINE, "bf16": lps.BF16_REFINE}[args.precision]
    eig = args.eig or ("fp32" if args.precision == "fp32" else "fp64")
    return {"precision": prec, "eig_precision": lps.EIG_FP64 if eig == "fp64" else lps.EIG_FP32}


def workload(frames, name="cardiac"):
    from paper_1411_6206_gb300 import phantom as P
    if name == "mix160":
        w = next(x for x in P.batched_mix(16, seed0=500) if (x.nx, x.nz, x.ncoil) == (160, 14, 16))
    else:
        w = P.CARDIAC if name == "cardiac" else P.PRECISION
    T = w.frames if frames is None else min(frames, w.frames)
    return w, T


def dc_kernel_name(w, tuned):
    """The data-consistency kernel a plan of workload w runs (default launch shapes or tuned)."""
    if tuned is not None and tuned.dc_variant in (1, 2):
        return "k_dc"
    if (w.ny, w.nz) == (128, 16):
        return "k_dc_reg"
    if (w.ny, w.nz) == (32, 8):
        return "k_dc_fixed"
    factors = w.ny % 8 == 0 and (w.ny <= 216 or w.ny in (224, 240, 256))
    return "k_dc_rows" if factors and w.nz <= 32 else "k_dc"


def dc_bytes_per_launch(w, m):
    """Algorithmic HBM bytes of one data-consistency launch of an iteration: coil maps and
    hybrid samples read; X_{k-1}, S_{k-1}, L_{k-1} and S_k read, X_k and L_k written
    (complex64)."""
    N = w.nx * w.ny * w.nz
    return N * (8 * w.ncoil + 48) + w.nx * w.ncoil * m * 8


def dc_flops_per_launch(w):
    """Nominal real flops of one data-consistency launch: per coil a forward and an inverse
    2D FFT of ny*nz points (5 n log2 n each), the coil multiply (6) and the conjugate-coil
    accumulate (8) per voxel, the reprojection L_k = (X - S) W in the prologue (8 nz per
    voxel) and the plane Gram epilogue (4 (nz + 1) per voxel)."""
    N = w.nx * w.ny * w.nz
    P = w.ny * w.nz
    return N * (w.ncoil * (10.0 * math.log2(P) + 14.0) + 8.0 * w.nz + 4.0 * (w.nz + 1))


def run_ours(args):
    import torch
    from paper_1411_6206_gb300 import lps, phantom as P

    ws, rank, local = dist()
    torch.cuda.set_device(local)
    if ws > 1:
        import torch.distributed as td
        td.init_process_group("nccl")
    w, T = workload(args.frames, args.workload)
    kw = plan_kw(args)
    dev = torch.device("cuda", local)
    stream = torch.cuda.Stream(device=dev)
    lib = lps.load()

    pr = P.problem(w, frames=T)
    coils = torch.from_numpy(np.ascontiguousarray(pr["coils"].astype(np.complex64))).to(dev)
    masks = [np.ascontiguousarray(m) for m in pr["masks"]]
    plan = lps.Plan(w.nx, w.ny, w.nz, w.ncoil, stream=stream, max_iters=w.iters, recursive=1, **kw)
    plan.set_coils(coils)
    # k-space of every frame by the library's forward operator, plus the generator's noise
    kdatas = []
    with torch.cuda.stream(stream):
        for t in range(T):
            n = plan.set_mask(masks[t])
            x = torch.from_numpy(np.ascontiguousarray(pr["x"][t].astype(np.complex64))).to(dev)
            kd = torch.empty((w.ncoil, n, w.nx), dtype=torch.complex64, device=dev)
            lps.forward(plan.handle, x, kd)
            kd += torch.from_numpy(pr["noise"][t].astype(np.complex64)).to(dev)
            kdatas.append(kd)
    stream.synchronize()
    tuned = None
    if args.workload == "mix160":
        plan.set_mask(masks[0])
        plan.set_data(kdatas[0])
        tuned = plan.autotune()
    nlines = [int(m.sum()) for m in masks]
    recon = torch.empty((T, w.nz, w.nx, w.ny), dtype=torch.complex64, device=dev)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    # the timed steps run the frame graph without in-graph events (they would serialise the
    # programmatic launches); the per-kernel times for the roofline come from a separate pass
    lps.set_profiling(plan.handle, False)

    def sequence(fev=None):
        plan.clear_prior()
        for t in range(T):
            if fev is not None:
                fev[t][0].record(stream)
            plan.set_mask(masks[t])
            plan.set_data(kdatas[t])
            plan.reconstruct_frame(recon=recon[t], stats=False)
            if fev is not None:
                fev[t][1].record(stream)

    ktimes = []
    step_ms = []
    frame_ms = []
    clocks = Clocks(local)
    for s in range(args.warmup + args.steps):
        timed = s >= args.warmup
        with torch.cuda.stream(stream):
            flush.zero_()
        stream.synchronize()
        if ws > 1:
            torch.distributed.barrier()
        torch.cuda.synchronize()
        if timed and s == args.warmup:
            clocks.start()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        fev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(T)]
        e0.record(stream)
        sequence(fev)
        e1.record(stream)
        stream.synchronize()
        if timed:
            step_ms.append(e0.elapsed_time(e1))
            frame_ms += [a.elapsed_time(b) for a, b in fev]
    clk = clocks.stop()
    torch.cuda.synchronize()
    if args.profile:
        # kernel-time pass (not part of `value`): CUDA events around every kernel of the graph
        lps.set_profiling(plan.handle, True)
        for s in range(2):
            with torch.cuda.stream(stream):
                flush.zero_()
            sequence()
            stream.synchronize()
            if s == 1:
                try:
                    ktimes.append(lps.get_kernel_times(plan.handle).as_dict())
                except lps.LpsError as e:
                    print(f"kernel times unavailable: {e}", file=sys.stderr)
        lps.set_profiling(plan.handle, False)
    total_ms = sum(step_ms)
    if ws > 1:
        t = torch.tensor([total_ms], device=dev)
        torch.distributed.all_reduce(t, op=torch.distributed.ReduceOp.MAX)
        total_ms = float(t.item())
    frames_done = ws * T * args.steps
    value = frames_done / (total_ms / 1e3)

    # end to end through the C ABI with host buffers: pinned k-space in, pinned recon out
    pin_k = [kd.cpu().pin_memory() for kd in kdatas]
    pin_out = torch.empty((T, w.nz, w.nx, w.ny), dtype=torch.complex64).pin_memory()
    plan_h = lps.Plan(w.nx, w.ny, w.nz, w.ncoil, stream=stream, max_iters=w.iters, recursive=1, **kw)
    plan_h.set_coils(coils)

    def seq_host():
        plan_h.clear_prior()
        for t in range(T):
            plan_h.set_mask(masks[t])
            plan_h.set_data(pin_k[t])
            plan_h.reconstruct_frame(recon=pin_out[t], stats=False)

    for _ in range(max(1, args.warmup)):
        seq_host()
    stream.synchronize()
    e2e_ms = []
    for _ in range(args.steps):
        with torch.cuda.stream(stream):
            flush.zero_()
        stream.synchronize()
        t0 = time.perf_counter()
        seq_host()
        stream.synchronize()
        e2e_ms.append((time.perf_counter() - t0) * 1e3)
    h2d = sum(int(k.numel()) * 8 + w.ny * w.nz for k in pin_k)
    d2h = T * w.nx * w.ny * w.nz * 8
    e2e_tot = sum(e2e_ms)
    if ws > 1:
        t = torch.tensor([e2e_tot], device=dev)
        torch.distributed.all_reduce(t, op=torch.distributed.ReduceOp.MAX)
        e2e_tot = float(t.item())
    e2e_value = ws * T * args.steps / (e2e_tot / 1e3)

    out = None
    if rank == 0:
        hbm, sm_max, src = peaks()
        alu_peak = SM_COUNT * FP32_LANES_PER_SM * 2 * sm_max * 1e6 / 1e12   # TFLOP/s
        roof = None
        # xfft, adjoint, haar-max, 3 per iteration, finalize, combine; the precision modes add the
        # tensor-core Gram (init + every iteration) and reprojection (every iteration)
        tc = args.precision != "fp32"
        launches_per_frame = (5 if tc else 3) * w.iters + 5 + (1 if tc else 0)
        if ktimes:
            # dominant kernel class over the timed steps
            tot = {k: sum(d[k]["ms"] for d in ktimes) for k in ktimes[0]}
            dom = max(tot, key=tot.get)
            n_l = sum(d[dom]["launches"] for d in ktimes)
            avg_ms = tot[dom] / max(n_l, 1)
            m_last = nlines[-1]
            if dom == "data_consistency":
                byts = dc_bytes_per_launch(w, m_last)
                gbs = byts / (avg_ms * 1e-3) / 1e9
                fl = dc_flops_per_launch(w) / (avg_ms * 1e-3) / 1e12
                frac_hbm, frac_alu = gbs / hbm, fl / alu_peak
                kname = dc_kernel_name(w, tuned)
                tr = profiled_traffic(f"{kname}_{args.workload}_{w.nx}x{w.ny}x{w.nz}x{w.ncoil}.txt")
                if frac_alu >= frac_hbm:
                    roof = {"bound": "alu", "achieved": round(fl, 3), "peak": round(alu_peak, 2),
                            "unit": "TFLOP/s", "frac": round(frac_alu, 4), "traffic": tr}
                else:
                    roof = {"bound": "hbm", "achieved": round(gbs, 1), "peak": hbm, "unit": "GB/s",
                            "frac": round(frac_hbm, 4), "traffic": tr}
                roof["kernel"] = f"{kname} (data consistency, step 4, with the reprojection of steps 1-2)"
                ws_mb = (w.nx * w.ny * w.nz * 8 * (w.ncoil + 6) + w.nx * w.ncoil * m_last * 8) / 1e6
                roof["regime"] = (f"working set ~{ws_mb:.0f} MB "
                                  + ("stays in the 129 MB L2 across iterations (flushed once per step): the "
                                     "fraction is of HBM peak, the kernel is latency-bound on L2-resident data"
                                     if ws_mb < 129 else "exceeds the 129 MB L2"))
                roof["algorithmic_bytes_per_launch"] = byts
                roof["alt"] = {"hbm_frac": round(frac_hbm, 4), "hbm_gbs": round(gbs, 1),
                               "alu_frac": round(frac_alu, 4), "alu_tflops": round(fl, 3)}
                roof["peak_source"] = (f"{src}: MEASURED_PEAKS.json hbm_gbs; FP32 = 152 SMs x 128 lanes x 2 "
                                       f"x sm_max_mhz")
            else:
                # one CTA by construction (an n x n problem): latency-bound; reported against the
                # whole-GPU FP32 peak, so the fraction is small by design
                fl = eig_flops_per_launch(w.nz) / (avg_ms * 1e-3) / 1e12
                roof = {"bound": "alu", "achieved": round(fl, 5), "peak": round(alu_peak, 2), "unit": "TFLOP/s",
                        "frac": round(fl / alu_peak, 6), "traffic": None,
                        "kernel": f"{dom} (single CTA; latency-bound)",
                        "peak_source": f"{src}: FP32 = 152 SMs x 128 lanes x 2 x sm_max_mhz"}
            roof["avg_launch_us"] = round(avg_ms * 1e3, 3)
            roof["share"] = {k: round(v / sum(tot.values()), 4) for k, v in tot.items()}
            nfr = len(ktimes)
            roof["us_per_launch"] = {k: round(1e3 * tot[k] / max(1, sum(d[k]["launches"] for d in ktimes)), 2)
                                     for k in tot}
            roof["kernel_ms_per_frame"] = round(sum(tot.values()) / nfr, 4)
        ms_step = total_ms / args.steps
        fl = sorted(frame_ms)
        out = {
            "metric": METRIC, "value": round(value, 2), "unit": "frames/s", "n_gpus": ws,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(ms_step, 4),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": {"fp32": "f32", "tf32": "tf32x2-split/f32", "bf16": "bf16x2-split/f32"}[args.precision],
            "data": "synthetic: seeded beating-heart phantom, smooth SoS coil maps, VD ky-kz masks, "
                    "CN noise; k-space made by the library's forward operator",
            "config": {"workload": f"{args.workload}-shaped recursive sequence {w.nx}x{w.ny}x{w.nz} x {T} frames, "
                                   f"{w.ncoil} coils, R={w.accel:g} (frame 1 at 50%), {w.iters} iterations/frame",
                       "nx": w.nx, "ny": w.ny, "nz": w.nz, "ncoil": w.ncoil, "frames": T, "iters": w.iters,
                       "mode": "plain (frame by frame, CUDA-graph replay per frame)",
                       "precision": args.precision, "eig": args.eig or ("fp32" if args.precision == "fp32" else "fp64"),
                       "l2": "256 MiB buffer written before every timed step (L2 flush)",
                       "parallelism": "independent sequence per GPU" if ws > 1 else "single GPU"},
            "frame_latency_ms": {"p50": round(float(np.percentile(fl, 50)), 4),
                                 "p99": round(float(np.percentile(fl, 99)), 4)},
            "roofline": roof,
            "e2e": {"value": round(e2e_value, 2), "unit": "frames/s", "h2d_bytes_per_step": h2d,
                    "d2h_bytes_per_step": d2h, "ms_per_step": round(e2e_tot / args.steps, 4)},
            "gpu_launches": launches_per_frame * T * args.steps,
            "clocks": clk,
        }
    plan_h.close()
    plan.close()
    if ws > 1:
        import torch.distributed as td
        td.barrier()
        td.destroy_process_group()
    return out, (w, T)


def cpu_baseline(args, w):
    """FP64 oracle on the host cores for a bounded sample of the workload (the first
    `cpu_frames` frames of the sequence, all iterations), and GPU parity on the same inputs.

    The GPU reconstructs the frames recursively; the oracle then reconstructs each frame from
    the same complex64 samples and the same prior (the support and singular values the GPU
    passed on from the previous frame). The threshold support rule makes the recursion
    discontinuous in coefficients that sit at the threshold, so each frame is compared given
    a common prior."""
    import scipy.fft as sfft
    import torch
    from oracle import lps_oracle as O
    from paper_1411_6206_gb300 import lps, phantom as P
    sys.path.insert(0, os.path.join(ROOT, "tests"))
    from abi_layout import bits_to_mallat

    F = max(1, args.cpu_frames)
    pr = P.problem(w, frames=F)
    coils64 = pr["coils"].astype(np.complex64)
    C128 = coils64.astype(np.complex128)
    datas = [(O.E(pr["x"][t], C128, pr["masks"][t]) + pr["noise"][t]).astype(np.complex64) for t in range(F)]
    plan = lps.Plan(w.nx, w.ny, w.nz, w.ncoil, max_iters=w.iters, recursive=1, **plan_kw(args))
    plan.set_coils(torch.from_numpy(coils64).cuda())
    gpu_out, priors = [], [None]
    out = torch.empty((w.nz, w.nx, w.ny), dtype=torch.complex64, device="cuda")
    sup = np.empty(plan.support_words(), np.uint32)
    sig = np.empty(w.nz)
    for t in range(F):
        plan.set_mask(pr["masks"][t])
        plan.set_data(torch.from_numpy(datas[t]).cuda())
        plan.reconstruct_frame(recon=out, support=sup, sigma=sig, stats=False)
        gpu_out.append(out.cpu().numpy())
        priors.append(O.Prior(support=bits_to_mallat(sup, w.nz, w.nx, w.ny, 3), sigma=sig.copy()))
    plan.close()
    p = O.Params(max_iters=w.iters)
    cores = os.cpu_count() or 1
    errs = []
    with sfft.set_workers(cores):
        t0 = time.perf_counter()
        for t in range(F):
            r = O.priori_ls(datas[t].astype(np.complex128), C128, pr["masks"][t], p, priors[t])
            errs.append(O.nrmse(gpu_out[t], r.recon))
        dt = time.perf_counter() - t0
    res = {"value": round(F / dt, 4), "unit": "frames/s", "cores": cores, "kind": "oracle",
           "sample": f"frames 1-{F} of the sequence, {w.iters} iterations each, FP64 NumPy/SciPy "
                     f"(scipy.fft workers = {cores})", "seconds": round(dt, 2)}
    return res, [round(e, 8) for e in errs]


def cpu_parity(small_job, prec_job):
    """Oracle comparisons of the GPU outputs kept by the small and precision studies (same
    complex64 samples, coil maps, masks and priors on both sides)."""
    import scipy.fft as sfft
    from oracle import lps_oracle as O
    sys.path.insert(0, os.path.join(ROOT, "tests"))
    from abi_layout import bits_to_mallat
    cores = os.cpu_count() or 1
    out = {}
    with sfft.set_workers(cores):
        if small_job is not None:
            w = small_job["w"]
            C = small_job["coils"].astype(np.complex128)
            p = O.Params(max_iters=w.iters)
            errs = []
            for t in range(2):
                pri = small_job["prior"][t]
                prior = None if pri is None else O.Prior(support=bits_to_mallat(pri[0], w.nz, w.nx, w.ny, 3),
                                                         sigma=pri[1])
                r = O.priori_ls(small_job["data"][t].astype(np.complex128), C, small_job["masks"][t], p, prior)
                errs.append(round(O.nrmse(small_job["recon"][t], r.recon), 8))
            out["small"] = errs
            f3 = small_job.get("frames3d")
            if f3 is not None:
                r = O.priori_ls(f3["data"].astype(np.complex128), f3["coils"].astype(np.complex128), f3["mask"],
                                O.Params(max_iters=w.iters, frame_slices=f3["fs"]))
                out["small_frames3d"] = round(O.nrmse(f3["recon"], r.recon), 8)
        if prec_job is not None:
            w = prec_job["w"]
            t0 = time.perf_counter()
            r = O.priori_ls(prec_job["data"].astype(np.complex128), prec_job["coils"].astype(np.complex128),
                            prec_job["mask"], O.Params(max_iters=w.iters))
            out["precision_oracle_s"] = round(time.perf_counter() - t0, 1)
            out["precision"] = {k: round(O.nrmse(v, r.recon), 9) for k, v in prec_job["recon"].items()}
    return out


def run_reference(args):
    """The FP64 oracle as the reference arm: each step reconstructs the next frame of the
    recursive sequence on the host cores."""
    import scipy.fft as sfft
    from oracle import lps_oracle as O
    from paper_1411_6206_gb300 import phantom as P

    ws, rank, _ = dist()
    if rank != 0:
        return None
    w, T = workload(args.frames, args.workload)
    nsteps = args.warmup + args.steps
    F = min(nsteps, w.frames)
    pr = P.problem(w, frames=F)
    coils = pr["coils"].astype(np.complex64).astype(np.complex128)
    datas = [(O.E(pr["x"][t], coils, pr["masks"][t]) + pr["noise"][t]).astype(np.complex64).astype(np.complex128)
             for t in range(F)]
    p = O.Params(max_iters=w.iters)
    cores = os.cpu_count() or 1
    prior = None
    times = []
    with sfft.set_workers(cores):
        for s in range(nsteps):
            t = s % F
            if t == 0:
                prior = None
            t0 = time.perf_counter()
            r = O.priori_ls(datas[t], coils, pr["masks"][t], p, prior)
            times.append(time.perf_counter() - t0)
            prior = O.Prior(support=r.support, sigma=r.sigma)
    tt = times[args.warmup:]
    value = len(tt) / sum(tt)
    fl = sorted(x * 1e3 for x in tt)
    return {
        "impl": "reference", "metric": METRIC, "value": round(value, 4), "unit": "frames/s",
        "n_gpus": ws, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": round(sum(tt) / len(tt) * 1e3, 2), "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic (same generator and seeds as the GPU arm)",
        "config": {"workload": f"{args.workload}-shaped recursive sequence {w.nx}x{w.ny}x{w.nz}, {w.ncoil} coils, "
                               f"R={w.accel:g}, {w.iters} iterations/frame; one frame per step",
                   "nx": w.nx, "ny": w.ny, "nz": w.nz, "ncoil": w.ncoil, "iters": w.iters},
        "frame_latency_ms": {"p50": round(float(np.percentile(fl, 50)), 2),
                             "p99": round(float(np.percentile(fl, 99)), 2)},
        "cpu_baseline": {"value": round(value, 4), "unit": "frames/s", "cores": cores, "kind": "oracle",
                         "sample": f"{len(tt)} frames of the recursive sequence, one per step"},
        "e2e": {"value": round(value, 4), "unit": "frames/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }


def gpu_problem(w, frames, lps, PG, P, dev, cycle=None):
    """Device-generated inputs of `frames` frames of workload w: coil maps, host masks and
    k-space made by the library's forward operator plus CN noise. With `cycle`, only that many
    distinct frames are made (the heart beats with a period of 8 frames)."""
    import torch
    coils = PG.coil_maps(w.nx, w.ny, w.nz, w.ncoil, w.seed, dev)
    masks = P.masks_for(w)
    hf = PG.HeartFrames(w, dev)
    fwd = lps.Plan(w.nx, w.ny, w.nz, w.ncoil, max_iters=1)
    fwd.set_coils(coils)
    n = frames if cycle is None else min(cycle, frames)
    out = []
    for t in range(n):
        m = masks[t % len(masks)]
        nl = fwd.set_mask(m)
        kd = torch.empty((w.ncoil, nl, w.nx), dtype=torch.complex64, device=dev)
        lps.forward(fwd.handle, hf.frame(t), kd)
        kd += PG.noise(w.ncoil, nl, w.nx, w.noise_sigma, w.seed * 1000 + t, dev)
        out.append((np.ascontiguousarray(m), kd))
    torch.cuda.synchronize()
    fwd.close()
    return coils, out


def serve_trace(n_sessions, rate, seconds, seed=5):
    """Poisson arrivals (seeded) of `rate` frames/s per session over `seconds`: [(time, session)]."""
    rng = np.random.default_rng(seed)
    trace = []
    for k in range(n_sessions):
        t = 0.0
        while True:
            t += rng.exponential(1.0 / rate)
            if t > seconds:
                break
            trace.append((t, k))
    trace.sort()
    return trace


def serve_once(lps, ws_, inputs, trace, single_stream, max_inflight):
    """One serving run over an arrival trace: every session's frames reconstructed recursively
    with its state resident; returns frames/s over the span and p50/p99 latency."""
    srv = lps.Server(150 * 10 ** 9, max_inflight=max_inflight, single_stream=single_stream, autotune=True)
    sids = [srv.open(lps.params_init(nx=w.nx, ny=w.ny, nz=w.nz, ncoil=w.ncoil, max_iters=w.iters,
                                     recursive=1), c) for w, (c, _) in zip(ws_, inputs)]
    nframe = [0] * len(sids)
    # warm-up: one frame per session (autotunes and captures the frame graphs)
    tk = [srv.submit(sid, *inputs[k][1][0], srv.now()) for k, sid in enumerate(sids)]
    for t in tk:
        srv.wait(t)
        srv.release(t)
    t0 = srv.now() + 0.05
    tickets = []
    for a, k in trace:
        while srv.now() < t0 + a:
            time.sleep(0.0001)
        fr = inputs[k][1][(1 + nframe[k]) % len(inputs[k][1])]
        nframe[k] += 1
        tickets.append(srv.submit(sids[k], fr[0], fr[1], t0 + a))
    lat, comp = [], []
    for t in tickets:
        l_, c_ = srv.wait(t)
        lat.append(l_)
        comp.append(c_)
        srv.release(t)
    span = max(comp) - (t0 + trace[0][0])
    srv.close()
    return {"frames_per_s": round(len(tickets) / span, 2),
            "p50_ms": round(1e3 * float(np.percentile(lat, 50)), 3),
            "p99_ms": round(1e3 * float(np.percentile(lat, 99)), 3),
            "frames": len(tickets)}


def run_served(args):
    """Serving study: sessions drawn from the uneven size mix, frames arriving as independent
    Poisson processes of 20 frames/s per session, reconstructed recursively with every
    session's state resident; served (per-session streams, no slot limit) against the plain
    path (every frame in arrival order on one stream) on the same arrival trace. With the
    sweep, the same at lower per-session rates (offered load below capacity, where p50/p99 are
    frame latencies rather than queue growth) and with a slot limit of 4 frames on the device."""
    from paper_1411_6206_gb300 import lps, phantom as P, phantom_gpu as PG
    import torch
    dev = torch.device("cuda", 0)
    ws_ = P.batched_mix(args.serve_sessions, seed0=500)
    inputs = [gpu_problem(w, w.frames, lps, PG, P, dev, cycle=8) for w in ws_]
    rate = 20.0
    trace = serve_trace(len(ws_), rate, args.serve_seconds)
    res = {mode: serve_once(lps, ws_, inputs, trace, mode == "plain", 0) for mode in ("served", "plain")}
    out = dict(res["served"])
    out["plain"] = res["plain"]
    # the same offered load over twice the arrival window: with capacity above the load the
    # latency percentiles stay put instead of growing with the queue
    long_s = 2.0 * args.serve_seconds
    out["long_window"] = dict(serve_once(lps, ws_, inputs, serve_trace(len(ws_), rate, long_s, seed=9), False, 0),
                              window_s=long_s)
    out.update({"sessions": len(ws_), "arrival_rate_per_session": rate, "offered_frames_per_s": rate * len(ws_),
                "window_s": args.serve_seconds, "hbm_budget_bytes": 150 * 10 ** 9,
                "sizes": [f"{w.nx}x{w.ny}x{w.nz}x{w.ncoil}c" for w in ws_],
                "how": "Poisson arrivals (seeded), latency = result ready (device event) - arrival, "
                       "server clock; plain = same trace, one stream in arrival order"})
    if not args.no_sweep:
        sweep = []
        for r, inflight in ((2.5, 0), (5.0, 0), (10.0, 0), (10.0, 4)):
            tr = serve_trace(len(ws_), r, min(args.serve_seconds, 4.0), seed=7)
            row = {"rate_per_session": r, "offered_frames_per_s": r * len(ws_), "max_inflight": inflight,
                   "served": serve_once(lps, ws_, inputs, tr, False, inflight)}
            if inflight == 0:
                row["plain"] = serve_once(lps, ws_, inputs, tr, True, 0)
            sweep.append(row)
        out["sweep"] = sweep
    return out


def run_batched(args):
    """Batched study: independent problems of uneven size (in-plane 64-160, 8-32 slices,
    10-30 frames, 4-16 coils, R 4-12), one graph launch per frame step after the autotuner
    picked each problem's launch shapes; against the same problems one frame graph at a time."""
    import torch
    from paper_1411_6206_gb300 import lps, phantom as P, phantom_gpu as PG
    dev = torch.device("cuda", 0)
    ws_ = P.batched_mix(args.batch_problems, seed0=400)
    inputs = [gpu_problem(w, w.frames, lps, PG, P, dev) for w in ws_]
    st = torch.cuda.Stream(device=dev)
    B = lps.Batch([lps.params_init(nx=w.nx, ny=w.ny, nz=w.nz, ncoil=w.ncoil, max_iters=w.iters, recursive=1)
                   for w in ws_], stream=st)
    for m, (c, fr) in zip(B.members, inputs):
        m.set_coils(c)
        m.set_mask(fr[0][0])
        m.set_data(fr[0][1])
    t_tune = time.perf_counter()
    B.autotune()
    t_tune = time.perf_counter() - t_tune
    T = max(w.frames for w in ws_)
    total = sum(w.frames for w in ws_)

    def sequence(batched):
        for m in B.members:
            m.clear_prior()
        for t in range(T):
            for i, w in enumerate(ws_):
                act = t < w.frames
                if batched:
                    B.set_active(i, act)
                if act:
                    B[i].set_mask(inputs[i][1][t][0])
                    B[i].set_data(inputs[i][1][t][1])
                    if not batched:
                        B[i].reconstruct_frame(stats=False)
            if batched:
                B.reconstruct()

    out = {}
    for mode in ("batched", "plain"):
        sequence(mode == "batched")      # warm-up (graph captures)
        st.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(st)
        sequence(mode == "batched")
        e1.record(st)
        st.synchronize()
        ms = e0.elapsed_time(e1)
        out[mode] = {"frames_per_s": round(total / (ms / 1e3), 2), "ms": round(ms, 2)}
    res = dict(out["batched"])
    res["plain"] = out["plain"]
    res.update({"problems": len(ws_), "frames": total, "frame_steps": T, "autotune_s": round(t_tune, 3),
                "how": "one graph launch per frame step over all problems (inactive members return at "
                       "once); plain = each problem's frame graph launched alone, in order"})
    # one data-consistency step (operator form) of all 64 problems: each member's own tuned kernel
    # as graph branches against one persistent launch over the descriptor table
    for i in range(len(ws_)):
        B.set_active(i, True)
    gen = torch.Generator(device=dev).manual_seed(3)
    Z = [torch.randn((w.nz, w.nx, w.ny), dtype=torch.complex64, device=dev, generator=gen) for w in ws_]
    X = [torch.empty_like(z) for z in Z]
    step = {}
    for name, pers in (("member_kernels", False), ("persistent", True)):
        B.data_consistency(Z, X, persistent=pers)
        step[name + "_ms"] = round(float(np.median([B.data_consistency(Z, X, persistent=pers) for _ in range(5)])), 3)
    step["how"] = ("step (4) of every problem once: each member's tuned kernel (factored rows "
                   "or runtime-sized) as parallel graph branches, against one persistent launch "
                   "whose CTAs take (problem, plane) items from a counter and run the runtime-sized body; "
                   "median of 5, device time")
    res["dc_step_all_problems"] = step
    B.close()
    return res


def forward_frames(lps, w, pr, T, dev, stream):
    """k-space of frames 0..T-1 of a problem by the library's forward operator, plus the
    generator's noise: coil maps on the device, host masks, device samples."""
    import torch
    coils = torch.from_numpy(np.ascontiguousarray(pr["coils"].astype(np.complex64))).to(dev)
    masks = [np.ascontiguousarray(m) for m in pr["masks"][:T]]
    fwd = lps.Plan(w.nx, w.ny, w.nz, w.ncoil, stream=stream, max_iters=1)
    fwd.set_coils(coils)
    kd = []
    with torch.cuda.stream(stream):
        for t in range(T):
            n = fwd.set_mask(masks[t])
            x = torch.from_numpy(np.ascontiguousarray(pr["x"][t].astype(np.complex64))).to(dev)
            k = torch.empty((w.ncoil, n, w.nx), dtype=torch.complex64, device=dev)
            lps.forward(fwd.handle, x, k)
            k += torch.from_numpy(pr["noise"][t].astype(np.complex64)).to(dev)
            kd.append(k)
    stream.synchronize()
    fwd.close()
    return coils, masks, kd


def run_small(args):
    """The 32 x 32 x 8 single-coil sequence (8 frames, 25% of the ky-kz lines, frame 1 at 50%,
    30 iterations): latency-bound, reported per frame. Returns the study and the GPU outputs of
    frames 1-2 (with the prior passed between them) for the CPU leg's oracle comparison."""
    import torch
    from paper_1411_6206_gb300 import lps, phantom as P
    w = P.SMALL
    T = w.frames
    pr = P.problem(w, frames=T)
    dev = torch.device("cuda", 0)
    st = torch.cuda.Stream(device=dev)
    coils, masks, kd = forward_frames(lps, w, pr, T, dev, st)
    pl = lps.Plan(w.nx, w.ny, w.nz, w.ncoil, stream=st, max_iters=w.iters, recursive=1)
    pl.set_coils(coils)
    out = torch.empty((T, w.nz, w.nx, w.ny), dtype=torch.complex64, device=dev)

    def seq():
        pl.clear_prior()
        for t in range(T):
            pl.set_mask(masks[t])
            pl.set_data(kd[t])
            pl.reconstruct_frame(recon=out[t], stats=False)

    for _ in range(3):
        seq()
    st.synchronize()
    ms = []
    for _ in range(10):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(st)
        seq()
        e1.record(st)
        st.synchronize()
        ms.append(e0.elapsed_time(e1))
    # frames 1-2 with the prior the GPU passes on, kept for the oracle comparison
    job = {"w": w, "coils": coils.cpu().numpy(), "masks": masks[:2], "data": [k.cpu().numpy() for k in kd[:2]],
           "recon": [], "prior": [None]}
    sup = np.empty(pl.support_words(), np.uint32)
    sig = np.empty(w.nz)
    one = torch.empty((w.nz, w.nx, w.ny), dtype=torch.complex64, device=dev)
    pl.clear_prior()
    for t in range(2):
        pl.set_mask(masks[t])
        pl.set_data(kd[t])
        pl.reconstruct_frame(recon=one, support=sup, sigma=sig, stats=False)
        job["recon"].append(one.cpu().numpy())
        job["prior"].append((sup.copy(), sig.copy()))
    pl.close()
    med = float(np.median(ms))
    res = {"workload": f"{w.nx}x{w.ny}x{w.nz} x {T} frames, {w.ncoil} coil, 25% of the ky-kz lines "
                       f"(frame 1 at 50%), {w.iters} iterations/frame, recursive",
           "us_per_frame": round(1e3 * med / T, 2), "frames_per_s": round(T / (med / 1e3), 1),
           "repeats": len(ms),
           "how": "CUDA events around the 8-frame sequence (median of 10, after 3 warm-up runs); the run "
                  "is launch- and latency-bound, so no roofline fraction is reported"}
    # the same 8 frames as one Casorati of volume columns (voxels x frames, layout "frames" with
    # 3D frames): one reconstruction of the segment from all frames' lines
    nzs = T * w.nz
    pf = lps.Plan(w.nx, w.ny, nzs, w.ncoil, stream=st, max_iters=w.iters, layout=lps.LAYOUT_FRAMES,
                  frame_slices=w.nz)
    pf.set_coils(torch.cat([coils] * T, dim=1).contiguous())
    mseg = np.ascontiguousarray(np.concatenate(masks, axis=0))
    pf.set_mask(mseg)
    dseg = torch.cat(list(kd), dim=1).contiguous()
    pf.set_data(dseg)
    seg = torch.empty((nzs, w.nx, w.ny), dtype=torch.complex64, device=dev)
    for _ in range(3):
        pf.reconstruct_frame(recon=seg, stats=False)
    ms3 = []
    for _ in range(10):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(st)
        pf.set_data(dseg)
        pf.reconstruct_frame(recon=seg, stats=False)
        e1.record(st)
        st.synchronize()
        ms3.append(e0.elapsed_time(e1))
    pf.close()
    med3 = float(np.median(ms3))
    res["frames3d"] = {"workload": f"{T} frames of {w.nx}x{w.ny}x{w.nz} as the Casorati columns "
                                   f"({w.nx * w.ny * w.nz} voxels x {T}), {w.iters} iterations",
                       "us_per_segment": round(1e3 * med3, 1), "frames_per_s": round(T / (med3 / 1e3), 1)}
    job["frames3d"] = {"coils": torch.cat([coils] * T, dim=1).cpu().numpy(), "mask": mseg,
                       "data": dseg.cpu().numpy(), "recon": seg.cpu().numpy(), "fs": w.nz}
    return res, job


def run_precision(args):
    """Precision study on the 192 x 192 x 32 sequence (12 coils, R = 10): frames/s per arithmetic
    (float32; tf32 and bf16 operands split hi + lo on the tensor cores with float32 accumulation
    and the float64 Rayleigh-Ritz eigen step), the tensor-core kernels' achieved bandwidth and
    algorithmic tensor rate, and NRMSE of frame 1 against the FP64 oracle."""
    import torch
    from paper_1411_6206_gb300 import lps, phantom as P
    w = P.PRECISION
    T = max(2, min(args.precision_frames, w.frames))
    pr = P.problem(w, frames=T)
    dev = torch.device("cuda", 0)
    st = torch.cuda.Stream(device=dev)
    coils, masks, kd = forward_frames(lps, w, pr, T, dev, st)
    job = {"w": w, "coils": coils.cpu().numpy(), "mask": masks[0], "data": kd[0].cpu().numpy(), "recon": {}}
    hbm, _, src = peaks()
    bf16_peak, tf32_peak, psrc = tensor_peaks()
    N = w.nx * w.ny * w.nz
    out = {"workload": f"{w.nx}x{w.ny}x{w.nz} x {T} frames, {w.ncoil} coils, R={w.accel:g} (frame 1 at 50%), "
                       f"{w.iters} iterations/frame, recursive"}
    recon = torch.empty((w.nz, w.nx, w.ny), dtype=torch.complex64, device=dev)
    for name in ("fp32", "tf32", "bf16"):
        prec = {"fp32": lps.FP32, "tf32": lps.TF32_REFINE, "bf16": lps.BF16_REFINE}[name]
        eig = lps.EIG_FP32 if name == "fp32" else lps.EIG_FP64
        pl = lps.Plan(w.nx, w.ny, w.nz, w.ncoil, stream=st, max_iters=w.iters, recursive=1, precision=prec,
                      eig_precision=eig)
        pl.set_coils(coils)

        def seq():
            pl.clear_prior()
            for t in range(T):
                pl.set_mask(masks[t])
                pl.set_data(kd[t])
                pl.reconstruct_frame(recon=recon, stats=False)

        seq()
        st.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(st)
        seq()
        e1.record(st)
        st.synchronize()
        ms = e0.elapsed_time(e1)
        lps.set_profiling(pl.handle, True)
        seq()
        st.synchronize()
        kt = lps.get_kernel_times(pl.handle).as_dict()
        lps.set_profiling(pl.handle, False)
        # frame 1 alone against the oracle
        pl.clear_prior()
        pl.set_mask(masks[0])
        pl.set_data(kd[0])
        pl.reconstruct_frame(recon=recon, stats=False)
        st.synchronize()
        job["recon"][name] = recon.cpu().numpy()
        pl.close()
        row = {"frames_per_s": round(T / (ms / 1e3), 2),
               "eig": "fp32 Jacobi" if name == "fp32" else "fp32 Jacobi + fp64 Rayleigh-Ritz",
               "us_per_launch": {k: round(1e3 * v["ms"] / max(1, v["launches"]), 2) for k, v in kt.items()
                                 if v["launches"]}}
        if name != "fp32":
            peak = bf16_peak if name == "bf16" else tf32_peak
            g_us = row["us_per_launch"].get("gram_tc")
            r_us = row["us_per_launch"].get("reproj_tc")
            # algorithmic work on the Casorati matrix (nx ny rows, nz columns): the Gram and the
            # reprojection are 8 (nx ny) nz^2 real flops each; the Gram reads X and S, the
            # reprojection reads X and S and writes L (complex64)
            fl = 8.0 * w.nx * w.ny * w.nz * w.nz
            row["gram_tc"] = {"us": g_us, "GB_s": round(2 * N * 8 / (g_us * 1e-6) / 1e9, 1),
                              "hbm_frac": round(2 * N * 8 / (g_us * 1e-6) / 1e9 / hbm, 4),
                              "algorithmic_TFLOP_s": round(fl / (g_us * 1e-6) / 1e12, 2),
                              "tensor_frac": round(fl / (g_us * 1e-6) / 1e12 / peak, 5)}
            row["reproj_tc"] = {"us": r_us, "GB_s": round(3 * N * 8 / (r_us * 1e-6) / 1e9, 1),
                                "hbm_frac": round(3 * N * 8 / (r_us * 1e-6) / 1e9 / hbm, 4),
                                "algorithmic_TFLOP_s": round(fl / (r_us * 1e-6) / 1e12, 2),
                                "tensor_frac": round(fl / (r_us * 1e-6) / 1e12 / peak, 5)}
        out[name] = row
    out["peaks"] = {"hbm_GB_s": hbm, "bf16_TFLOP_s": bf16_peak, "tf32_TFLOP_s": tf32_peak,
                    "source": f"{src}; tensor: {psrc}"}
    out["how"] = ("frames/s: CUDA events around the sequence after one warm-up sequence; kernel times from a "
                  "separate pass with events around every kernel; tensor_frac = algorithmic flops of the "
                  "contraction over the dense peak of the operand type (the split operands add products "
                  "executed on the pipe)")
    return out, job


def plan_variants(variants, kernel):
    """The cardiac-shaped sequence on plans that differ in lps_params fields only: frames/s
    (median of 3 sequences, L2 flushed before each) and the time per launch of one kernel
    class (a profiling pass), per variant."""
    import torch
    from paper_1411_6206_gb300 import lps, phantom as P
    w = P.CARDIAC
    T = w.frames
    pr = P.problem(w, frames=T)
    dev = torch.device("cuda", 0)
    st = torch.cuda.Stream(device=dev)
    coils, masks, kd = forward_frames(lps, w, pr, T, dev, st)
    out = {}
    recon = torch.empty((T, w.nz, w.nx, w.ny), dtype=torch.complex64, device=dev)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    for name, kw in variants:
        pl = lps.Plan(w.nx, w.ny, w.nz, w.ncoil, stream=st, max_iters=w.iters, recursive=1, **kw)
        pl.set_coils(coils)

        def seq():
            pl.clear_prior()
            for t in range(T):
                pl.set_mask(masks[t])
                pl.set_data(kd[t])
                pl.reconstruct_frame(recon=recon[t], stats=False)

        seq()
        ms = []
        for _ in range(3):
            with torch.cuda.stream(st):
                flush.zero_()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(st)
            seq()
            e1.record(st)
            st.synchronize()
            ms.append(e0.elapsed_time(e1))
        lps.set_profiling(pl.handle, True)
        seq()
        st.synchronize()
        kt = lps.get_kernel_times(pl.handle).as_dict()[kernel]
        words = np.empty(pl.support_words(), np.uint32)
        lps.get_support(pl.handle, words, None)
        pl.close()
        out[name] = {"frames_per_s": round(T / (float(np.median(ms)) / 1e3), 2),
                     kernel + "_us_per_launch": round(1e3 * kt["ms"] / max(1, kt["launches"]), 2),
                     "support_fraction_last_frame": round(
                         float(np.unpackbits(words.view(np.uint8)).sum()) / (32 * words.size), 4)}
    return out


def run_coils_fp16(args):
    """The cardiac-shaped sequence with the coil maps stored in half precision (LPS_COILS_FP16):
    frames/s and the data-consistency kernel's time per launch against float32 maps."""
    from paper_1411_6206_gb300 import lps
    out = plan_variants((("fp32", dict(coil_format=lps.COILS_FP32)), ("fp16", dict(coil_format=lps.COILS_FP16)),
                         ("fp16_maps_and_samples", dict(coil_format=lps.COILS_FP16, data_format=lps.DATA_FP16))),
                        "data_consistency")
    out["how"] = ("same inputs, float32 maps and samples given to every plan (the fp16 plans round them); the "
                  "effect of the rounding on the reconstruction is measured by tests/test_gpu_coils_fp16.py and "
                  "tests/test_gpu_data_fp16.py")
    return out


def run_haar3(args):
    """The cardiac-shaped sequence with the 3D Haar (wavelet_dims = 3) against the per-slice 2D
    Haar: frames/s, the sparse-step kernel's time per launch and the support fraction."""
    out = plan_variants((("haar2d", dict(wavelet_dims=2)), ("haar3d", dict(wavelet_dims=3))), "sparse_step")
    out["how"] = ("same inputs and iteration count; the 3D variant adds the z pass through shared memory "
                  "to the sparse-step kernel")
    return out


def run_window(args):
    """Sliding temporal window over a 2D + time stream (128 x 128 slice of the cardiac-shaped
    phantom, 8 coils, R = 8 per frame, window W = 16 frames, 50 iterations per window): output
    frames/s and the latency of each pushed frame (its window's reconstruction)."""
    import torch
    from paper_1411_6206_gb300 import lps, phantom as P
    from paper_1411_6206_gb300.window import SlidingWindow
    T, W, nx, ny, nc = 40, 16, 128, 128, 8
    w = P.Workload("stream", nx, ny, 1, nc, T, 50, 8.0, 31, phantom="heart")
    x = P.phantom_sequence(w)[:, 0]
    dev = torch.device("cuda", 0)
    st = torch.cuda.Stream(device=dev)
    c1 = torch.from_numpy(np.ascontiguousarray(P.coil_maps(nx, ny, 1, nc, 37)[:, 0].astype(np.complex64))).to(dev)
    fwd = lps.Plan(nx, ny, 1, nc, stream=st, fft_z=0, max_iters=1)
    fwd.set_coils(c1[:, None].contiguous())
    frames = []
    with torch.cuda.stream(st):
        for t in range(T):
            m = P.vd_mask(ny, 1, ny // 8, 4, 500 + t, 0)
            n = fwd.set_mask(m)
            k = torch.empty((nc, n, nx), dtype=torch.complex64, device=dev)
            lps.forward(fwd.handle, torch.from_numpy(np.ascontiguousarray(x[t][None].astype(np.complex64))).to(dev), k)
            k += torch.from_numpy(P.noise(nc, n, nx, 1e-3, 600 + t).astype(np.complex64)).to(dev)
            frames.append((m[0], k))
    st.synchronize()
    fwd.close()
    out = {}
    for rep in range(2):   # the first pass captures the window graph
        sw = SlidingWindow(lps, nx, ny, nc, W, c1, stream=st, max_iters=50)
        lat = []
        with torch.cuda.stream(st):
            e0 = torch.cuda.Event(enable_timing=True)
            e0.record(st)
            for t in range(T):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record(st)
                r = sw.push(*frames[t])
                b.record(st)
                if r is not None:
                    lat.append((a, b))
            e1 = torch.cuda.Event(enable_timing=True)
            e1.record(st)
        st.synchronize()
        ms = [a.elapsed_time(b) for a, b in lat]
        out = {"frames_out": len(ms), "frames_per_s": round(len(ms) / (e0.elapsed_time(e1) / 1e3), 2),
               "p50_ms": round(float(np.percentile(ms, 50)), 4), "p99_ms": round(float(np.percentile(ms, 99)), 4)}
        sw.close()
    out["workload"] = (f"2D + time stream {nx}x{ny}, {nc} coils, {ny // 8} ky lines per frame, window {W} frames, "
                       f"50 iterations per window, {T} frames pushed")
    out["how"] = "CUDA events around each push (set_mask, set_data, frame graph) on the plan's stream"
    return out


def run_fig3(args):
    """Synthetic analogue of the paper's Fig. 3 (Sec. 4): mean PSNR against the ground-truth
    phantom over frames 2-20 of the cardiac-shaped sequence, plain L+S (every frame without a
    prior) against Priori L+S (the recursion of Sec. 3), at several undersampling factors;
    frame 1 is sampled at 50% in both."""
    import dataclasses
    import torch
    from paper_1411_6206_gb300 import lps, phantom as P
    dev = torch.device("cuda", 0)
    st = torch.cuda.Stream(device=dev)
    rows = []
    for R in (4, 6, 8, 10, 12):
        w = dataclasses.replace(P.CARDIAC, accel=float(R))
        T = w.frames
        pr = P.problem(w, frames=T)
        coils, masks, kd = forward_frames(lps, w, pr, T, dev, st)
        row = {"R": R, "sampling": round(1.0 / R, 4)}
        for mode in ("plain", "priori"):
            pl = lps.Plan(w.nx, w.ny, w.nz, w.ncoil, stream=st, max_iters=w.iters, recursive=1)
            pl.set_coils(coils)
            out = torch.empty((w.nz, w.nx, w.ny), dtype=torch.complex64, device=dev)
            ps = []
            for t in range(T):
                if mode == "plain" or t == 0:
                    pl.clear_prior()
                pl.set_mask(masks[t])
                pl.set_data(kd[t])
                pl.reconstruct_frame(recon=out, stats=False)
                st.synchronize()
                if t == 0:
                    continue
                x = pr["x"][t]
                mse = float(np.mean(np.abs(out.cpu().numpy().astype(np.complex128) - x) ** 2))
                ps.append(10.0 * np.log10(float(np.max(np.abs(x))) ** 2 / mse))
            pl.close()
            row[f"psnr_{mode}_db"] = round(float(np.mean(ps)), 3)
        row["gain_db"] = round(row["psnr_priori_db"] - row["psnr_plain_db"], 3)
        rows.append(row)
    return {"rows": rows,
            "how": "cardiac-shaped phantom family (128x128x16, 8 coils, beating heart on a rank-4 background), "
                   "per-frame VD ky-kz masks at 1/R of the lines (frame 1 at 50%), 50 iterations per frame; "
                   "PSNR = 10 log10(max|x|^2 / mean|recon - x|^2) against the phantom, mean over frames 2-20; "
                   "plain = the prior cleared before every frame (plain L+S with its own lambdas)"}


def tensor_peaks():
    """Dense bf16 peak (measured burst figure) and the tf32 peak derived from it by the nominal
    1.1 / 2.25 ratio."""
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(p) as f:
            d = json.load(f)
        bf = float(d["bf16_tflops"])
        return bf, round(bf * 1.1 / 2.25, 1), "measured bf16 (MEASURED_PEAKS.json), tf32 = bf16 x 1.1/2.25"
    except Exception:
        return 1900.0, round(1900.0 * 1.1 / 2.25, 1), "fallback bf16 1.9 PFLOP/s, tf32 = bf16 x 1.1/2.25"


def main():
    args = parse()
    if args.impl == "reference":
        out = run_reference(args)
        if out is not None:
            print(json.dumps(out), flush=True)
        return
    out, (w, T) = run_ours(args)
    ws, rank, _ = dist()
    if rank == 0:
        if ws == 1 and not args.no_served:
            out["served"] = run_served(args)
        if ws == 1 and not args.no_batched:
            out["batched"] = run_batched(args)
        small_job = prec_job = None
        if ws == 1 and not args.no_small:
            out["small"], small_job = run_small(args)
        if ws == 1 and not args.no_precision:
            out["precision"], prec_job = run_precision(args)
        if ws == 1 and not args.no_fig3:
            out["fig3"] = run_fig3(args)
        if ws == 1 and not args.no_small:
            out["coils_fp16"] = run_coils_fp16(args)
            out["haar3d"] = run_haar3(args)
            out["window"] = run_window(args)
        if ws == 1 and not args.no_cpu_baseline:
            cb, nr = cpu_baseline(args, w)
            out["cpu_baseline"] = cb
            out["nrmse_vs_oracle"] = {"max": max(nr), "per_frame": nr,
                                      "how": "GPU recursive frames vs the FP64 oracle on the same "
                                             "samples and the same prior; bound 1e-3"}
            par = cpu_parity(small_job, prec_job)
            if "small" in par:
                out["small"]["nrmse_vs_oracle"] = par["small"]
            if "small_frames3d" in par:
                out["small"]["frames3d"]["nrmse_vs_oracle"] = par["small_frames3d"]
            if "precision" in par:
                for k, v in par["precision"].items():
                    out["precision"][k]["nrmse_frame1_vs_oracle"] = v
                out["precision"]["oracle_frame1_s"] = par["precision_oracle_s"]
        print(json.dumps(out), flush=True)


if __name__ == "__main__":
    main()
