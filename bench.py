#!/usr/bin/env python
"""Benchmark: HDCR time-to-1e-10 against plain FP64 CR, and the fine-stencil bandwidth.

Workload (the two-level FP64 configuration): 16^4 lattice, Ls = 16, synthetic
links U = exp(i eps H) with eps = 0.5, M5 = 1.8, mf = 0.01, one Gaussian
source; nvec = 24 subspace vectors on 4^4 blocks (a 4^4 coarse lattice).

One step = one pass of the whole hot path on that input:
  subspace (Chebyshev low-pass filter of 12 Gaussian noise fields, Gamma5 split,
  FP64 block Gram-Schmidt) -> little Dirac operator (FP64 build, dense inverse)
  -> HDCR solve (FP64 flexible GCR, V-cycle with the order-10 Chebyshev
  smoother and the exact coarse solve) to a true residual of 1e-10
  -> the gauge-link force of the solution.
``value`` is seconds per step (lower is better).  Beside it the JSON line
reports plain FP64 CR to the same tolerance on the same GPU, the FP32-inner
variant, the FP32 stencil bandwidth against the measured HBM peak, the
roofline of the dominant kernel, the CPU oracle baseline, the end-to-end time
through host buffers, SM clocks during the timed region and the number of
library kernels launched.

Usage: python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
                       [--workload two-level|precision|batching|table1]
Under torchrun each rank runs an independent replica (the solve does not
shard across GPUs here); rank 0 prints one JSON line.

The default workload is the one above.  Two more print their own line:
``precision`` (24^3 x 48 x 16, eps = 0.5, mf = 0.005: FP32 stencil and its
FP16-storage variant, the coarse operator with nvec = 32 on the tensor cores,
the mixed-precision solve with an FP64 outer iteration to 1e-10) and
``batching`` (16^3 x 32 x 16, the 12 spin-colour point sources solved at once
with the graph-captured V-cycle, against 12 single solves; the coarse operator
with nvec = 48) and ``table1`` (the setting of the paper's Table 1: 16^3 x 32 x 16
at valence mass 0.001, red-black CGNE against HDCR, setup and solve apart).
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

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "HDCR time-to-1e-10 vs plain FP64 CR on same GB300; Γ5Ddwf GB/s as % HBM peak"
L_FINE = (16, 16, 16, 16)
LS = 16
EPS = 0.5
M5 = 1.8
MF = 0.01
NVEC = 24
BLOCK = (4, 4, 4, 4)
SEED_GAUGE, SEED_SRC, SEED_NOISE = 1001, 2001, 3001
# filter order 200: on this workload orders 200, 250, 300 and 400 give the same
# solve (18 outer iterations, 814 fine applications, for four noise seeds), 175
# needs 20 and 150 stalls; cut 0.3 (0.25 needs 24 iterations, 0.5 at order 200 stalls)
FILTER = dict(kind="chebyshev", order=200, lam_cut=0.3, lam_max=8.0)
# FGCR restart 24: longer than the ~17 outer iterations the solve takes, so the
# search space is never thrown away (restart 8: 18 iterations, 814 applications;
# 24 or 32: 17, 767)
SOLVE = dict(tol=1e-10, restart=24, smoother="chebyshev", smoother_order=10, cheb_lo=1.0, cheb_hi=64.0,
             coarse_solver="dense", max_outer=200)
# Algorithmic floating-point operations per 5d site of one application of H (real
# adds and multiplies, an FMA counted as 2): the Wilson hopping term in its
# standard count, 8 hops x (12 spin projection + 132 SU(3) x half-spinor + 24
# accumulation) - 24 (the first hop initialises the sum) = 1320; the -1/2 scale of
# the hop sum (24), the (5 - M5) diagonal (24), adding the two (24) and the two
# fifth-dimension hops P_-psi(s+1), P_+psi(s-1) (12 complex subtractions, 24): 1416.
# Gamma5 and the R5 reflection are signs and a permutation (free).
FLOPS_PER_SITE = 1320 + 4 * 24


# algorithmic bytes per 5d site of one application (read psi, write H psi, links / Ls)
def bytes_per_site(real_bytes: int, Ls: int) -> float:
    return 2 * 12 * 2 * real_bytes + 4 * 9 * 2 * real_bytes / Ls


# DRAM traffic of one FP64 / FP32 / FP16-storage stencil launch at 16^4 x 16 from ncu, with the hash of
# the stencil sources it was measured on (reported as null once the sources change)
NCU_TRAFFIC = {"f64": 571.81e6, "f32": 202.18e6, "h16": 106.18e6, "src_hash": "6cf224fdd680fc72"}


def stencil_src_hash() -> str:
    h = hashlib.sha256()
    for f in ("dwf_stencil.cuh", "dwf.cu", "dwf_fx.cu", "dwf_fx.cuh", "fx_device.cuh", "dwf_x2.cu", "dwf_x2.cuh", "dwf_h16.cu",
              "hdcr_internal.cuh"):
        with open(os.path.join(ROOT, "paper_1611_06944_gb300", "csrc", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def peaks() -> dict:
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            d = json.load(f)
        return {"hbm_gbs": float(d["hbm_gbs"]), "source": "measured"}
    except Exception:
        return {"hbm_gbs": 6800.0, "source": "fallback"}


# ------------------------------------------------------------------ clocks
class ClockSampler:
    """nvidia-smi samples of SM clock and throttle reasons while running."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu: int):
        self.gpu = gpu
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits", "-lms", "200",
                 "-i", str(self.gpu)], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except Exception:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self) -> dict:
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                mx.append(float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": sorted(reasons), "samples": len(sm)}


# ------------------------------------------------------------------ distributed
def dist_setup():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch.distributed as dist
        backend = "nccl" if _cuda() else "gloo"
        dist.init_process_group(backend=backend)
    return world, rank, local


def _cuda() -> bool:
    import torch
    return torch.cuda.is_available()


def aggregate(elapsed_s: float, units: int, world: int) -> dict:
    """Whole-job figures from this rank's timed seconds: the max over ranks, and the
    total units processed by all ranks (each rank runs ``units`` steps)."""
    t = elapsed_s
    if world > 1:
        import torch
        import torch.distributed as dist
        dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
        x = torch.tensor([elapsed_s], dtype=torch.float64, device=dev)
        dist.all_reduce(x, op=dist.ReduceOp.MAX)
        t = float(x.item())
    total_units = units * world
    return {"max_seconds": t, "total_units": total_units, "seconds_per_unit": t / total_units}


def barrier(world: int):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


# ------------------------------------------------------------------ workload
def make_inputs(device: str):
    import numpy as np
    import torch

    import synth
    lat_L = L_FINE
    U = synth.gauge_field(lat_L, EPS, SEED_GAUGE)
    plaq = synth.plaquette(U)
    Uh = torch.from_numpy(np.ascontiguousarray(U.reshape(4, -1, 3, 3)))
    b = synth.gaussian_fermion(lat_L, LS, SEED_SRC)
    noise = synth.gaussian_fermion(lat_L, LS, SEED_NOISE, count=NVEC // 2)
    # natural (…, Lt, Lz, Ly, Lx, Ls, 4, 3) -> library layout (…, V4, 12, Ls)
    def pack(a):
        lead = a.shape[:-7]
        return np.ascontiguousarray(np.swapaxes(a.reshape(lead + (-1, LS, 12)), -1, -2))
    bh = torch.from_numpy(pack(b))
    nh = torch.from_numpy(pack(noise))
    return Uh, bh, nh, plaq


def hdcr_step(hd, lat, U, b, noise, inner="f64"):
    """One pass of the hot path; returns (x, stats dict)."""
    import torch
    tdt = torch.complex128 if inner == "f64" else torch.complex64
    sub = hd.build_subspace(lat, U, noise, M5, MF, BLOCK, filter_dtype=torch.complex64, store_dtype=tdt,
                            **FILTER)
    co = hd.build_coarse_op(sub, U, M5, MF, op_dtype=tdt, fp32_build=tdt == torch.complex128)
    hd.coarse_invert(co)
    x, st = hd.hdcr_solve(co, U, b, inner_dtype=tdt, **SOLVE)
    F = hd.gauge_force(lat, x, hd.apply_gamma5_r5(lat, x))
    co.close()
    sub.close()
    return x, F, st


def step_breakdown(hd, lat, U, b, noise) -> dict:
    """Wall time of each phase of one step, synchronising between phases (outside the timed region)."""
    import torch
    out = {}

    def tick(name, t0):
        torch.cuda.synchronize()
        out[name] = round(time.perf_counter() - t0, 4)
        return time.perf_counter()

    torch.cuda.synchronize()
    t = time.perf_counter()
    sub = hd.build_subspace(lat, U, noise, M5, MF, BLOCK, filter_dtype=torch.complex64,
                            store_dtype=torch.complex128, **FILTER)
    t = tick("subspace_s", t)
    co = hd.build_coarse_op(sub, U, M5, MF, op_dtype=torch.complex128, fp32_build=True)
    t = tick("coarse_op_s", t)
    hd.coarse_invert(co)
    t = tick("coarse_invert_s", t)
    x, st = hd.hdcr_solve(co, U, b, inner_dtype=torch.complex128, **SOLVE)
    t = tick("solve_s", t)
    hd.gauge_force(lat, x, hd.apply_gamma5_r5(lat, x))
    tick("force_s", t)
    co.close()
    sub.close()
    return out


def run_ours(args, world, rank, local):
    import numpy as np
    import torch

    import paper_1611_06944_gb300 as hd
    torch.cuda.set_device(local)
    dev = f"cuda:{local}"
    lat = hd.Lattice(L_FINE, LS, 1)
    Uh, bh, nh, plaq = make_inputs(dev)
    U, b, noise = Uh.to(dev), bh.to(dev), nh.to(dev)
    stream = torch.cuda.current_stream()
    for _ in range(args.warmup):
        hdcr_step(hd, lat, U, b, noise)
    torch.cuda.synchronize()
    barrier(world)
    torch.cuda.synchronize()
    clocks = ClockSampler(local)
    clocks.start()
    hd.stencil_timer(True)
    n0 = hd.launch_count()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    stats = []
    for _ in range(args.steps):
        x, F, st = hdcr_step(hd, lat, U, b, noise)
        stats.append(st)
    e1.record(stream)
    torch.cuda.synchronize()
    launches = hd.launch_count() - n0
    clk = clocks.stop()
    st64 = hd.stencil_timer_read(torch.complex128)
    st64c = hd.stencil_timer_read(torch.complex128, fused_cheb=True)
    st32 = hd.stencil_timer_read(torch.complex64)
    hd.stencil_timer(False)
    barrier(world)
    elapsed = e0.elapsed_time(e1) / 1e3
    agg = aggregate(elapsed, args.steps, world)
    if rank != 0:
        return None
    # ---------------------------------------------------------- comparisons (outside the timed region)
    x_cr = torch.zeros_like(b)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    x_cr, st_cr = hd.cr_solve(lat, U, b, M5, MF, tol=1e-10, max_iter=100000)
    torch.cuda.synchronize()
    t_cr = time.perf_counter() - t0
    # the paper's own comparison solver (Section 5, Table 1): red-black CGNE, FP64
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    x_rb, st_rb = hd.cgne_rb_solve(lat, U, b, M5, MF, tol=1e-10, max_iter=100000)
    torch.cuda.synchronize()
    t_rb = time.perf_counter() - t0
    del x_rb
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    _, _, st_mixed = hdcr_step(hd, lat, U, b, noise, inner="f32")
    torch.cuda.synchronize()
    t_mixed = time.perf_counter() - t0
    sol_diff = float(torch.linalg.vector_norm(x - x_cr) / torch.linalg.vector_norm(x_cr))
    phases = step_breakdown(hd, lat, U, b, noise)
    # FP32 stencil bandwidth (the second half of the metric)
    U32, b32 = U.to(torch.complex64), b.to(torch.complex64)
    y32 = torch.empty_like(b32)
    for _ in range(3):
        hd.apply_g5dwf(lat, U32, b32, M5, MF, out=y32)
    torch.cuda.synchronize()
    hd.stencil_timer(True)
    for _ in range(50):
        hd.apply_g5dwf(lat, U32, b32, M5, MF, out=y32)
    torch.cuda.synchronize()
    s32 = hd.stencil_timer_read(torch.complex64)
    hd.stencil_timer(False)
    h16 = _stencil_rate(hd, lat, U32, hd.encode_h16(lat, b), h16=True)
    h16["traffic"] = NCU_TRAFFIC["h16"] if NCU_TRAFFIC["src_hash"] == stencil_src_hash() else None
    pk = peaks()
    bps32 = bytes_per_site(4, LS)
    gbs32 = s32["sites"] * bps32 / (s32["ms"] * 1e-3) / 1e9
    # ---------------------------------------------------------- roofline of the dominant kernel
    same_src = NCU_TRAFFIC["src_hash"] == stencil_src_hash()
    ms64 = st64["ms"] / max(st64["launches"], 1)
    sites64 = st64["sites"] / max(st64["launches"], 1)
    achieved = FLOPS_PER_SITE * sites64 / (ms64 * 1e-3) / 1e12
    share64 = ms64 * st64["all_launches"] / (elapsed * 1e3)   # every FP64 launch at the timed average
    # the FP64 applications that carry the fused smoother step (1416 + 144 flops per site)
    ms64c = st64c["ms"] / max(st64c["launches"], 1)
    share64c = ms64c * st64c["all_launches"] / (elapsed * 1e3)
    fp64_peak = hd.probe_fma_rate(torch.complex128)            # measured on this GPU, this run
    bps64 = bytes_per_site(8, LS)
    gbs64 = sites64 * bps64 / (ms64 * 1e-3) / 1e9
    roofline = {"bound": "hbm", "kernel": "g5dwf FP64 in fixed point (H = Gamma5 D_dwf, with the operand's encoding "
                                          "where the solve has not encoded it already)",
                "achieved": round(gbs64, 1), "peak": pk["hbm_gbs"], "unit": "GB/s",
                "frac": round(gbs64 / pk["hbm_gbs"], 4), "traffic": NCU_TRAFFIC["f64"] if same_src else None,
                "bytes_per_site": bps64, "flops_per_site": FLOPS_PER_SITE, "tflops": round(achieved, 4),
                "fp64_fma_tflops": round(fp64_peak, 4), "avg_launch_ms": round(ms64, 4),
                "share_of_step": round(share64, 3), "peak_source": pk["source"],
                "with_fused_smoother_step": {
                    "kernel": "the same with one Chebyshev recurrence step in its epilogue",
                    "launches_per_step": round(st64c["all_launches"] / max(args.steps, 1), 1),
                    "avg_launch_ms": round(ms64c, 4), "share_of_step": round(share64c, 3),
                    "tflops": round((FLOPS_PER_SITE + 144) * st64c["sites"] / max(st64c["launches"], 1)
                                    / max(ms64c * 1e-3, 1e-12) / 1e12, 4)},
                "peak_note": "the kernel does its products on the integer pipe and is limited by "
                             "instruction issue, not by memory; fp64_fma_tflops is the FP64 pipe's measured rate "
                             "(hdcr_probe_fma_rate, FMA = 2 flops), which bounded the operator as FP64 FMAs"}
    roofline_fp32 = {"bound": "hbm", "kernel": "g5dwf FP32 (H = Gamma5 D_dwf)", "achieved": round(gbs32, 1),
                     "peak": pk["hbm_gbs"], "unit": "GB/s", "frac": round(gbs32 / pk["hbm_gbs"], 4),
                     "traffic": NCU_TRAFFIC["f32"] if same_src else None, "bytes_per_site": bps32,
                     "peak_source": pk["source"]}
    # ---------------------------------------------------------- e2e through host buffers
    e2e = run_e2e(hd, lat, Uh, bh, nh, stream)
    solve_mv = stats[-1]["fine_matvecs"] + stats[-1]["fine_matvecs_lo"]
    mv_step = step_matvecs(solve_mv)
    cpu = cpu_baseline(args, mv_step, solve_mv) if world == 1 else None
    line = {
        "metric": METRIC,
        "value": round(agg["seconds_per_unit"], 4),
        "unit": "s",
        "n_gpus": world,
        "steps": args.steps,
        "warmup": args.warmup,
        "ms_per_step": round(agg["max_seconds"] * 1e3 / args.steps, 2),
        "higher_is_better": False,
        "scaling": "weak",
        "vs_baseline": None,
        "dtype": "f64",
        "data": "synthetic",
        "config": {
            "workload": "two-level FP64: 16^4 x 16 DWF, eps=0.5, M5=1.8, mf=0.01, 1 Gaussian source, "
                        "nvec=24, 4^4 blocks (4^4 coarse)",
            "plaquette": round(plaq, 4),
            "step": f"Chebyshev-filter subspace (order {FILTER['order']}, FP32 filter, FP64 Gram-Schmidt) + coarse op "
                    "(FP32-exact tensor-core build, stored FP64) + FP32 dense coarse inverse + FP64 HDCR solve "
                    "(FP64 smoother and outer GCR) to 1e-10 + gauge force",
            "l2": "inputs larger than L2 (201 MB per FP64 field)",
            "parallelism": f"replicas x{world}",
        },
        "hdcr": {"outer_iters": stats[-1]["iters"], "fine_matvecs": stats[-1]["fine_matvecs"],
                 "coarse_solves": stats[-1]["coarse_matvecs"], "true_resid": stats[-1]["true_resid"],
                 "solve_s": round(stats[-1]["t_total"], 4), "smoother_s": round(stats[-1]["t_smoother"], 4),
                 "coarse_s": round(stats[-1]["t_coarse"], 4)},
        "step_phases": phases,
        "plain_fp64_cr": {"seconds": round(t_cr, 4), "iters": st_cr["iters"], "true_resid": st_cr["true_resid"],
                          "speedup_of_hdcr_step": round(t_cr / agg["seconds_per_unit"], 3),
                          "solution_rel_diff": sol_diff},
        "red_black_cgne_fp64": {"seconds": round(t_rb, 4), "iters": st_rb["iters"],
                                "hop_applications": st_rb["fine_matvecs"], "true_resid": st_rb["true_resid"],
                                "speedup_of_hdcr_step": round(t_rb / agg["seconds_per_unit"], 3),
                                "speedup_of_hdcr_solve": round(t_rb / stats[-1]["t_total"], 3)},
        "hdcr_fp32_inner": {"seconds": round(t_mixed, 4), "outer_iters": st_mixed["iters"],
                            "true_resid": st_mixed["true_resid"], "fine_matvecs_f64": st_mixed["fine_matvecs"],
                            "fine_matvecs_f32": st_mixed["fine_matvecs_lo"]},
        "g5dwf_fp32": {"GBs": round(gbs32, 1), "frac_of_hbm": round(gbs32 / pk["hbm_gbs"], 4),
                       "hbm_peak_gbs": pk["hbm_gbs"], "peak_source": pk["source"],
                       "bytes_per_site": bps32, "avg_launch_us": round(s32["ms"] / s32["launches"] * 1e3, 2),
                       "traffic": NCU_TRAFFIC["f32"] if same_src else None},
        "g5dwf_fp16_storage": h16,
        "roofline": roofline,
        "roofline_fp32": roofline_fp32,
        "e2e": e2e,
        "gpu_launches": int(launches),
        "clocks": clk,
    }
    if cpu is not None:
        line["cpu_baseline"] = cpu
    return line


def run_e2e(hd, lat, Uh, bh, nh, stream) -> dict:
    """The same step through the C ABI with HOST buffers: the pinned host links, noise
    and source are handed to the library's entry points (hdcr_build_subspace,
    hdcr_build_coarse_op, hdcr_solve), which stage them through device buffers
    themselves, and the solution, Gamma5 x and the force come back into host buffers
    (hdcr_solve, hdcr_apply_gamma5_r5, hdcr_gauge_force); every copy is inside the
    timed region."""
    import torch
    Up, bp, npin = Uh.pin_memory(), bh.pin_memory(), nh.pin_memory()
    xh = torch.zeros_like(bh).pin_memory()
    wh = torch.empty_like(bh).pin_memory()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    sub = hd.build_subspace(lat, Up, npin, M5, MF, BLOCK, filter_dtype=torch.complex64,
                            store_dtype=torch.complex128, **FILTER)
    co = hd.build_coarse_op(sub, Up, M5, MF, op_dtype=torch.complex128, fp32_build=True)
    hd.coarse_invert(co)
    st = hd.hdcr_solve_into(co, Up, bp, xh, inner_dtype=torch.complex128, **SOLVE)
    hd.apply_gamma5_r5(lat, xh, wh)
    F = hd.gauge_force(lat, xh, wh)
    e1.record(stream)
    torch.cuda.synchronize()
    co.close()
    sub.close()
    t = e0.elapsed_time(e1) / 1e3
    fb = bh.numel() * 16
    # in: links three times (subspace, coarse operator, solve), the noise, and the source,
    # the initial guess, x for Gamma5 and x, w for the force; out: x, Gamma5 x and F
    h2d = 3 * Uh.numel() * 16 + nh.numel() * 16 + 5 * fb
    d2h = 2 * fb + F.numel() * 16
    return {"value": round(t, 4), "unit": "s", "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(d2h),
            "path": "C ABI with pinned host buffers (staged by the library)", "status": st["status"],
            "true_resid": st["true_resid"]}


# applications of H in one solve of the step as measured on GB300 (17 outer iterations)
SOLVE_MATVECS = 767


def step_matvecs(solve_mv: int) -> int:
    """Applications of H in one step, the unit the oracle's time is scaled by: the
    subspace filter (NVEC/2 fields x 2 per order), the coarse build (about one per
    basis vector) and the solve."""
    return NVEC // 2 * 2 * FILTER["order"] + NVEC + solve_mv


def _oracle_worker(job: tuple):
    """One process of the CPU baseline: applications of the oracle's H on the lattice
    (L, Ls) for about ``seconds``; returns the seconds per application."""
    L, Ls, seconds = job
    import synth
    from oracle import dwf
    U = synth.gauge_field(L, EPS, SEED_GAUGE)
    b = synth.gaussian_fermion(L, Ls, SEED_SRC)
    dwf.apply_H(U, b, M5, MF)  # warm-up
    n, t0 = 0, time.perf_counter()
    while n < 1 or (time.perf_counter() - t0 < seconds and n < 4):
        dwf.apply_H(U, b, M5, MF)
        n += 1
    return (time.perf_counter() - t0) / n


def oracle_sample(workers: int, seconds: float = 8.0) -> dict:
    """Seconds per oracle application of H at 16^4 x 16 measured on ``workers`` host cores
    at once (processes started with spawn, so a CUDA context in this process is not
    inherited) and on one core alone."""
    import multiprocessing as mp
    ctx = mp.get_context("spawn")
    job = (L_FINE, LS, seconds)
    with ctx.Pool(workers) as pool:
        par = pool.map(_oracle_worker, [job] * workers)
    single = _oracle_worker(job)
    return {"per_apply_parallel_s": statistics.median(par), "per_apply_single_s": single, "workers": workers}


def step_oracle_seconds(smp: dict, solve_mv: int) -> float:
    """The oracle's time for one step on ``workers`` cores, from the sampled rates: the
    NVEC/2 filtered noise fields are independent (one per core, 2 x order applications
    each), the coarse build applies H to the NVEC basis vectors independently, the solve
    is one sequential chain of applications.  A lower bound: the oracle's Gram-Schmidt,
    inverse and BLAS are not counted."""
    w = smp["workers"]
    fields = NVEC // 2
    filt = -(-fields // w) * 2 * FILTER["order"] * smp["per_apply_parallel_s"]
    build = -(-NVEC // w) * smp["per_apply_parallel_s"]
    return filt + build + solve_mv * smp["per_apply_single_s"]


def cpu_baseline(args, mv_step: int, solve_mv: int) -> dict:
    """The FP64 numpy oracle on this host's cores: a bounded sample of applications of H
    on the full lattice, run by one process per core at once and by one alone, scaled to
    one step (step_oracle_seconds)."""
    w = max(1, min(16, _host_cores()))
    smp = oracle_sample(w)
    v = step_oracle_seconds(smp, solve_mv)
    return {"value": round(v, 2), "unit": "s", "cores": w, "kind": "oracle",
            "sample": f"applications of the oracle's H at 16^4x16 on {w} processes at once "
                      f"({smp['per_apply_parallel_s']:.2f} s each) and on one alone "
                      f"({smp['per_apply_single_s']:.2f} s), scaled to a step: the {NVEC // 2} filtered noise "
                      f"fields in parallel (2 x {FILTER['order']} applications each), the {NVEC} basis "
                      f"vectors of the coarse build in parallel, the solve's {solve_mv} applications in sequence "
                      f"(a lower bound: Gram-Schmidt, inverse and BLAS not counted)",
            "threads_note": f"numpy, one process per core (spawn); {_host_cores()} cores available"}


def _cpu_seconds() -> float:
    import resource
    r = resource.getrusage(resource.RUSAGE_SELF)
    return r.ru_utime + r.ru_stime


def _threads_used(c0: float, wall: float) -> int:
    """Threads the oracle kept busy on average since c0 (CPU seconds / wall seconds)."""
    return max(1, round((_cpu_seconds() - c0) / max(wall, 1e-9)))


def _host_cores() -> int:
    try:
        return len(os.sched_getaffinity(0))
    except Exception:
        return os.cpu_count() or 1


def run_reference(args, world, rank):
    """The oracle on the host cores, each step a bounded sample of the workload: the
    applications of H of one step (step_oracle_seconds) timed on one process per core and
    on one alone, scaled to the step."""
    if rank != 0:
        return None
    w = max(1, min(16, _host_cores()))
    for _ in range(args.warmup):
        oracle_sample(w, seconds=1.0)
    vals = []
    for _ in range(args.steps):
        smp = oracle_sample(w, seconds=2.0)
        vals.append(step_oracle_seconds(smp, SOLVE_MATVECS))
    v = round(statistics.median(vals), 2)
    return {"impl": "reference", "metric": METRIC, "value": v, "unit": "s", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(v * 1e3, 2),
            "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic",
            "config": {"workload": "two-level FP64: 16^4 x 16 DWF, eps=0.5, M5=1.8, mf=0.01, nvec=24, 4^4 blocks"},
            "cpu_baseline": {"value": v, "unit": "s", "cores": w, "kind": "oracle",
                             "sample": f"each step: oracle applications of H at 16^4x16 on {w} processes at once "
                                       f"and on one alone, scaled to one HDCR step ({NVEC // 2} filter fields and "
                                       f"{NVEC} coarse-build vectors in parallel, {SOLVE_MATVECS} solve "
                                       f"applications in sequence)"},
            "e2e": {"value": v, "unit": "s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}


# ------------------------------------------------------------------ further workloads
def _sync_time(fn):
    import torch
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    r = fn()
    torch.cuda.synchronize()
    return r, time.perf_counter() - t0


def _stencil_rate(hd, lat, U32, x, h16=False, reps=20) -> dict:
    """Event-timed FP32 (or FP16-storage) applications of H: us per launch and GB/s of
    algorithmic bytes (spinor in + out, links once per 4d site)."""
    import torch
    y = torch.empty_like(x)
    nf = (x.numel() // (52 * lat.V5)) if h16 else hd._nfields(lat, x, "x")
    apply = (lambda: hd.apply_g5dwf_h16(lat, U32, x, M5, MF, out=y)) if h16 else \
        (lambda: hd.apply_g5dwf(lat, U32, x, M5, MF, out=y))
    for _ in range(3):
        apply()
    torch.cuda.synchronize()
    hd.stencil_timer(True)
    for _ in range(reps):
        apply()
    torch.cuda.synchronize()
    t = hd.stencil_timer_read("h16" if h16 else torch.complex64)
    hd.stencil_timer(False)
    us = t["ms"] / t["launches"] * 1e3
    per_site = (2 * 52 if h16 else 2 * 96) + 4 * 72 / lat.Ls / nf
    gbs = lat.V5 * nf * per_site / (us * 1e-6) / 1e9
    pk = peaks()["hbm_gbs"]
    return {"us": round(us, 2), "GBs": round(gbs, 1), "frac_of_hbm": round(gbs / pk, 4), "bytes_per_site": per_site,
            "fields": nf}


def _coarse_rebuild(hd, sub, U, mf, fast: bool, mv_ms: float, reps=3) -> dict:
    import torch
    hd.build_coarse_op(sub, U, M5, mf, op_dtype=torch.complex64, fast=fast).close()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(reps):
        hd.build_coarse_op(sub, U, M5, mf, op_dtype=torch.complex64, fast=fast).close()
    e1.record()
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / reps
    return {"ms": round(ms, 2), "fine_matvecs": round(ms / mv_ms, 1),
            "projection": "single-pass TF32" if fast else "three-pass TF32 (FP32-exact)"}


def run_precision(args, world, rank, local):
    """24^3 x 48 x 16, eps = 0.5, mf = 0.005: the mixed-precision form."""
    import torch

    import paper_1611_06944_gb300 as hd
    import synth
    torch.cuda.set_device(local)
    L, Ls, eps, mf, nvec = (24, 24, 24, 48), 16, 0.5, 0.005, 32
    lat = hd.Lattice(L, Ls, 1)
    Uh = synth.gauge_field(L, eps, 1002)
    plaq = synth.plaquette(Uh)
    U = torch.from_numpy(Uh.reshape(4, -1, 3, 3).copy()).cuda()
    del Uh
    U32 = U.to(torch.complex64)
    b = synth.device_gaussian(1, lat.V5, 2002)[0].reshape(lat.V4, 12, Ls).contiguous()
    noise = synth.device_gaussian(nvec // 2, lat.V5, 3002).reshape(nvec // 2, lat.V4, 12, Ls).contiguous()
    x32 = b.to(torch.complex64)
    f32 = _stencil_rate(hd, lat, U32, x32)
    h16 = _stencil_rate(hd, lat, U32, hd.encode_h16(lat, b), h16=True)
    # order 600 with the cut at 0.1 (orders 300 and cuts 0.3 left the solve stalled near 1e-4
    # on this lattice; the paper's own filter is O(500-900))
    filt = dict(kind="chebyshev", order=600, lam_cut=0.1, lam_max=8.0, filter_dtype=torch.complex64,
                store_dtype=torch.complex64)
    # 6^4 blocks (coarse 4^3 x 8, 16384 unknowns): the dense coarse inverse applies.  With
    # 4^4 blocks (82944 unknowns, beyond the dense inverse) the coarse solve is the recursive
    # one (measured below); coarse CR to 1e-6 also converges but needs ~3000 CR iterations
    # per coarse solve
    block = (6, 6, 6, 6)
    solve = dict(tol=1e-10, restart=8, smoother="chebyshev", smoother_order=10, cheb_lo=1.0, cheb_hi=64.0,
                 coarse_solver="dense", max_outer=300, inner_dtype=torch.complex64)
    phases = {}

    def step():
        sub, t_sub = _sync_time(lambda: hd.build_subspace(lat, U, noise, M5, mf, block, **filt))
        co, t_co = _sync_time(lambda: hd.build_coarse_op(sub, U, M5, mf, op_dtype=torch.complex64, fast=True))
        _, t_inv = _sync_time(lambda: hd.coarse_invert(co))
        (x, st), t_solve = _sync_time(lambda: hd.hdcr_solve(co, U, b, **solve))
        phases.update(subspace_s=round(t_sub, 3), coarse_op_s=round(t_co, 4), coarse_invert_s=round(t_inv, 3),
                      solve_s=round(t_solve, 3))
        co.close()
        return sub, x, st

    for _ in range(args.warmup):
        sub, x, st = step()
        sub.close()
    clocks = ClockSampler(local)
    clocks.start()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(args.steps):
        sub, x, st = step()
        if _ + 1 < args.steps:
            sub.close()
    e1.record()
    torch.cuda.synchronize()
    clk = clocks.stop()
    elapsed = e0.elapsed_time(e1) / 1e3 / args.steps
    rebuild = {"6^4 blocks": {"fast": _coarse_rebuild(hd, sub, U, mf, True, f32["us"] * 1e-3),
                              "exact": _coarse_rebuild(hd, sub, U, mf, False, f32["us"] * 1e-3)}}
    sub.close()
    # the 4^4 blocks of the paper's other workloads (6^3 x 12 coarse lattice, 82,944 coarse unknowns:
    # beyond the dense inverse, so the coarse solve is the recursive one with a third level on
    # 2^4 blocks of the coarse lattice)
    sub4, t_sub4 = _sync_time(lambda: hd.build_subspace(lat, U, noise, M5, mf, BLOCK, **filt))
    rebuild["4^4 blocks"] = {"fast": _coarse_rebuild(hd, sub4, U, mf, True, f32["us"] * 1e-3),
                             "exact": _coarse_rebuild(hd, sub4, U, mf, False, f32["us"] * 1e-3)}
    co4, t_co4 = _sync_time(lambda: hd.build_coarse_op(sub4, U, M5, mf, op_dtype=torch.complex64, fast=True))
    cvec = sub4.Vc * nvec                        # one coarse vector
    half2 = 32                                   # 64 level-2 vectors
    n2 = synth.device_gaussian(half2, -(-cvec // 12), 3012)[:, :cvec].reshape(half2, sub4.Vc, nvec).contiguous()
    _, t_l2 = _sync_time(lambda: hd.build_level2(co4, n2, (2, 2, 2, 2), smooth_iters=200, cycle_smooth=16))
    solve4 = dict(solve, coarse_solver="recursive", coarse_tol=1e-6, coarse_max=100)
    (x4, st4), t_solve4 = _sync_time(lambda: hd.hdcr_solve(co4, U, b, **solve4))
    recursive = {"blocks": list(BLOCK), "coarse_unknowns": sub4.Vc * nvec, "level2_blocks": [2, 2, 2, 2],
                 "level2_unknowns": sub4.Vc // 16 * 2 * half2, "subspace_s": round(t_sub4, 3),
                 "coarse_op_s": round(t_co4, 4), "level2_build_s": round(t_l2, 3), "solve_s": round(t_solve4, 3),
                 "outer_iters": st4["iters"], "coarse_gcr_iters": st4["coarse_matvecs"],
                 "true_resid": st4["true_resid"], "fine_matvecs_f32": st4["fine_matvecs_lo"],
                 "fine_matvecs_f64": st4["fine_matvecs"]}
    co4.close()
    sub4.close()
    return {
        "metric": METRIC, "workload_kind": "precision", "value": round(elapsed, 3), "unit": "s",
        "n_gpus": world, "steps": args.steps, "warmup": args.warmup, "higher_is_better": False,
        "dtype": "f32 inner / f64 outer", "data": "synthetic (links on the host, noise and source drawn on the device)",
        "config": {"workload": "precision form: 24^3x48 x 16 DWF, eps=0.5, M5=1.8, mf=0.005, 1 Gaussian source, "
                               "nvec=32, 6^4 blocks (4^3x8 coarse)", "plaquette": round(plaq, 4),
                   "step": "Chebyshev-filter subspace (order 600, FP32) + coarse op (TF32 tensor cores, one pass) + "
                           "dense coarse inverse + FP64 flexible GCR with FP32 V-cycle (Chebyshev smoother) to 1e-10"},
        "phases": phases,
        "hdcr": {"outer_iters": st["iters"], "true_resid": st["true_resid"], "fine_matvecs_f64": st["fine_matvecs"],
                 "fine_matvecs_f32": st["fine_matvecs_lo"], "coarse_matvecs": st["coarse_matvecs"]},
        "g5dwf_fp32": f32, "g5dwf_fp16_storage": h16, "coarse_rebuild_nvec32": rebuild,
        "recursive_coarse_solve_4x4_blocks": recursive, "clocks": clk,
    }


def run_batching(args, world, rank, local):
    """16^3 x 32 x 16, the 12 spin-colour point sources at once."""
    import torch

    import paper_1611_06944_gb300 as hd
    import synth
    torch.cuda.set_device(local)
    L, Ls, eps, mf, nvec = (16, 16, 16, 32), 16, 0.5, 0.01, 48
    lat = hd.Lattice(L, Ls, 1)
    Uh = synth.gauge_field(L, eps, 1003)
    plaq = synth.plaquette(Uh)
    U = torch.from_numpy(Uh.reshape(4, -1, 3, 3).copy()).cuda()
    U32 = U.to(torch.complex64)
    # the 12 point sources at x = 0, s = 0 (component 3 spin + colour), in the library layout
    B = torch.zeros(12, lat.V4, 12, Ls, dtype=torch.complex128, device="cuda")
    for i in range(12):
        B[i, 0, i, 0] = 1.0
    noise = synth.device_gaussian(nvec // 2, lat.V5, 3003).reshape(nvec // 2, lat.V4, 12, Ls).contiguous()
    f32_1 = _stencil_rate(hd, lat, U32, noise[0].to(torch.complex64).contiguous())
    f32_12 = _stencil_rate(hd, lat, U32, noise[:12].to(torch.complex64).contiguous())
    sub, t_sub = _sync_time(lambda: hd.build_subspace(lat, U, noise, M5, mf, BLOCK, kind="chebyshev", order=300,
                                                      lam_cut=0.3, lam_max=8.0, filter_dtype=torch.complex64,
                                                      store_dtype=torch.complex64))
    rebuild = {"fast": _coarse_rebuild(hd, sub, U, mf, True, f32_1["us"] * 1e-3),
               "exact": _coarse_rebuild(hd, sub, U, mf, False, f32_1["us"] * 1e-3)}
    co, t_co = _sync_time(lambda: hd.build_coarse_op(sub, U, M5, mf, op_dtype=torch.complex64, fast=True))
    _, t_inv = _sync_time(lambda: hd.coarse_invert(co))
    kw = dict(tol=1e-10, restart=8, max_outer=300, inner_dtype=torch.complex64)
    for _ in range(args.warmup):
        hd.hdcr_solve_multi(co, U, B, graph=True, **kw)
    clocks = ClockSampler(local)
    clocks.start()
    n0 = hd.launch_count()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(args.steps):
        X, stats = hd.hdcr_solve_multi(co, U, B, graph=True, **kw)
    e1.record()
    torch.cuda.synchronize()
    clk = clocks.stop()
    launches = (hd.launch_count() - n0) / args.steps
    t_multi = e0.elapsed_time(e1) / 1e3 / args.steps
    _, t_eager = _sync_time(lambda: hd.hdcr_solve_multi(co, U, B, graph=False, **kw))

    def singles():
        its = []
        for i in range(12):
            _, s1 = hd.hdcr_solve(co, U, B[i].contiguous(), smoother="chebyshev", coarse_solver="dense", **kw)
            its.append(s1["iters"])
        return its

    its, t_single = _sync_time(singles)
    co.close()
    sub.close()
    return {
        "metric": METRIC, "workload_kind": "batching", "value": round(t_multi, 3), "unit": "s",
        "n_gpus": world, "steps": args.steps, "warmup": args.warmup, "higher_is_better": False,
        "dtype": "f32 inner / f64 outer", "data": "synthetic (links on the host, noise on the device)",
        "config": {"workload": "batching form: 16^3x32 x 16 DWF, eps=0.5, M5=1.8, mf=0.01, 12 spin-colour point "
                               "sources, nvec=48, 4^4 blocks (4^3x8 coarse)", "plaquette": round(plaq, 4),
                   "step": "12-source HDCR solve to 1e-10 in lockstep (FP32 V-cycle replayed from a CUDA graph, "
                           "FP64 outer), dense coarse inverse"},
        "setup": {"subspace_s": round(t_sub, 3), "coarse_op_s": round(t_co, 4), "coarse_invert_s": round(t_inv, 3)},
        "multi": {"seconds": round(t_multi, 3), "outer_iters": stats[0]["iters"],
                  "max_true_resid": max(s["true_resid"] for s in stats), "launches_per_solve": int(launches),
                  "eager_seconds": round(t_eager, 3)},
        "single_solves": {"seconds": round(t_single, 3), "iters": its},
        "g5dwf_fp32": {"nrhs1": f32_1, "nrhs12": f32_12}, "coarse_rebuild_nvec48": rebuild, "clocks": clk,
    }


# the subspace filter of the Table 1 setting (valence mf = 0.001).  Measured with
# the FP32 V-cycle: order 300 at cut 0.2 reaches 1e-10 in 20 outer iterations after
# 2.4 s of setup, 400 / 0.2 in 21 after 2.9 s, 600 / 0.1 in 19 after 3.8 s; 400 / 0.1,
# 300 / 0.1, 300 / 0.15 and 200 / 0.2 stall above 1e-4 in 300 iterations
TABLE1_FILTER = dict(kind="chebyshev", order=300, lam_cut=0.2, lam_max=8.0)


def run_table1(args, world, rank, local):
    """The setting of the paper's Table 1 on synthetic links: 16^3 x 32 x 16, valence
    mf = 0.001, one Gaussian source; red-black CGNE (FP64) against HDCR (Chebyshev
    filter subspace, FP32 V-cycle, FP64 outer), setup and solve reported apart as in
    the table.  The paper's 16 vectors left HDCR stalled near 1e-3 on these links;
    32 are used.  A solve that does not reach 1e-10 is reported with its status."""
    import torch

    import paper_1611_06944_gb300 as hd
    import synth
    torch.cuda.set_device(local)
    L, Ls, eps, mf, nvec = (16, 16, 16, 32), 16, 0.5, 0.001, 32
    lat = hd.Lattice(L, Ls, 1)
    Uh = synth.gauge_field(L, eps, 1003)
    plaq = synth.plaquette(Uh)
    U = torch.from_numpy(Uh.reshape(4, -1, 3, 3).copy()).cuda()
    b = synth.device_gaussian(1, lat.V5, 2003)[0].reshape(lat.V4, 12, Ls).contiguous()
    noise = synth.device_gaussian(nvec // 2, lat.V5, 3003).reshape(nvec // 2, lat.V4, 12, Ls).contiguous()
    xr = torch.empty_like(b)

    def cgne():
        st = hd._lib.hdcr_solve_stats()
        g, p = lat.c_geom(), hd._params(M5, mf)
        hd._L.hdcr_cgne_rb_solve(hd.C_ref(g), hd.C_ref(p), U.data_ptr(), b.data_ptr(), xr.data_ptr(), 1e-10, 40000,
                                 hd.C_ref(st), torch.cuda.current_stream().cuda_stream)
        return st.as_dict()

    st_rb, t_rb = _sync_time(cgne)
    del xr

    def setup():
        sub, t_sub = _sync_time(lambda: hd.build_subspace(lat, U, noise, M5, mf, BLOCK, **TABLE1_FILTER,
                                                          filter_dtype=torch.complex64, store_dtype=torch.complex64))
        co, t_co = _sync_time(lambda: hd.build_coarse_op(sub, U, M5, mf, op_dtype=torch.complex64, fast=True))
        _, t_inv = _sync_time(lambda: hd.coarse_invert(co))
        return sub, co, t_sub, t_co, t_inv

    if args.warmup > 0:  # one untimed setup: first-use costs (stencil tuner, cuBLAS handle, kernel attributes)
        sub, co, *_ = setup()
        co.close()
        sub.close()
    sub, co, t_sub, t_co, t_inv = setup()
    kw = dict(tol=1e-10, restart=8, max_outer=300, inner_dtype=torch.complex64)
    x = torch.zeros_like(b)
    for _ in range(args.warmup):
        x.zero_()
        hd.hdcr_solve_into(co, U, b, x, **kw)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(args.steps):
        x.zero_()
        st = hd.hdcr_solve_into(co, U, b, x, **kw)
    e1.record()
    torch.cuda.synchronize()
    t_solve = e0.elapsed_time(e1) / 1e3 / args.steps
    co.close()
    sub.close()
    setup = t_sub + t_co + t_inv
    return {
        "metric": METRIC, "workload_kind": "table1", "value": round(t_solve, 3), "unit": "s",
        "n_gpus": world, "steps": args.steps, "warmup": args.warmup, "higher_is_better": False,
        "dtype": "f32 inner / f64 outer (HDCR), f64 (CGNE)", "data": "synthetic (links on the host, noise and "
                                                                    "source drawn on the device)",
        "config": {"workload": "Table 1 setting: 16^3x32 x 16 DWF, eps=0.5, M5=1.8, valence mf=0.001, 1 Gaussian "
                               "source, nvec=32, 4^4 blocks (4^3x8 coarse)", "plaquette": round(plaq, 4),
                   "subspace": f"Chebyshev filter of order {TABLE1_FILTER['order']}, cut {TABLE1_FILTER['lam_cut']}, "
                               "FP32"},
        "red_black_cgne_fp64": {"seconds": round(t_rb, 3), "iters": st_rb["iters"], "status": st_rb["status"],
                                "hop_applications": st_rb["fine_matvecs"], "true_resid": st_rb["true_resid"]},
        "hdcr": {"solve_s": round(t_solve, 3), "setup_s": round(setup, 3), "status": st["status"],
                 "setup": {"subspace_s": round(t_sub, 3), "coarse_op_s": round(t_co, 4), "coarse_invert_s": round(t_inv, 3)},
                 "outer_iters": st["iters"], "fine_matvecs_f32": st["fine_matvecs_lo"],
                 "fine_matvecs_f64": st["fine_matvecs"], "true_resid": st["true_resid"],
                 "speedup_of_solve_over_cgne": round(t_rb / t_solve, 3),
                 "speedup_of_setup_plus_solve_over_cgne": round(t_rb / (t_solve + setup), 3)},
    }


def run_differentiation(args, world, rank, local):
    """8^3 x 16, Ls = 8: loss Re(eta^dag x), x = hdcr_solve(U, b) differentiated by the
    backward (adjoint HDCR solve with the subspace rebuilt + gauge force), in complex128
    and complex64.  value = seconds of one forward + backward in complex128; the
    gradient's error against the FP64 oracle gradient (tests/golden, written by the
    oracle alone) is reported for both precisions."""
    import numpy as np
    import torch

    import paper_1611_06944_gb300 as hd
    import synth
    torch.cuda.set_device(local)
    with open(os.path.join(ROOT, "tests", "golden", "grad_8x8x8x16_ls8.json")) as f:
        gd = json.load(f)
    L, Ls, mf = tuple(gd["lattice"]), gd["Ls"], gd["mf"]
    lat = hd.Lattice(L, Ls, gd["bc_t"])
    U = synth.gauge_field(L, gd["eps"], gd["seeds"]["U"]).reshape(4, -1, 3, 3)

    def planes(a):
        return np.ascontiguousarray(np.swapaxes(a.reshape(-1, Ls, 12), -1, -2))

    b = planes(synth.gaussian_fermion(L, Ls, gd["seeds"]["b"]))
    eta = planes(synth.gaussian_fermion(L, Ls, gd["seeds"]["eta"]))
    noise = torch.from_numpy(planes(synth.gaussian_fermion(L, Ls, 6003, count=8)).reshape(8, -1, 12, Ls)).cuda()
    want = np.array([[complex(r, i) for r, i in v] for _, _, v in gd["links"]])
    out = {}
    for name, dt, tol in (("c128", torch.complex128, 1e-12), ("c64", torch.complex64, 1e-7)):
        def step():
            Ut = torch.from_numpy(U).cuda().to(dt).requires_grad_(True)
            bt = torch.from_numpy(b).cuda().to(dt).requires_grad_(True)
            x = hd.solve_autograd(lat, Ut, bt, noise, gd["M5"], mf, (4, 4, 4, 4),
                                  filter_kw=dict(kind="chebyshev", order=100),
                                  solve_kw=dict(tol=tol, max_outer=500))
            loss = torch.vdot(torch.from_numpy(eta).cuda().to(dt).reshape(-1), x.reshape(-1)).real
            loss.backward()
            return Ut.grad
        for _ in range(args.warmup):
            step()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(args.steps):
            g = step()
        e1.record()
        torch.cuda.synchronize()
        gU = g.cpu().numpy().astype(np.complex128)
        got = np.array([gU[mu, x4].reshape(-1) for mu, x4, _ in gd["links"]])
        err = float(np.linalg.norm(got - want) / np.linalg.norm(want))
        out[name] = {"seconds_fwd_bwd": round(e0.elapsed_time(e1) / 1e3 / args.steps, 4),
                     "grad_rel_err_vs_fp64_oracle": err, "solve_tol": tol,
                     "sample": f"{len(gd['links'])} links (9 entries each) of dL/dU"}
    return {"metric": METRIC, "workload_kind": "differentiation", "value": out["c128"]["seconds_fwd_bwd"],
            "unit": "s", "n_gpus": world, "steps": args.steps, "warmup": args.warmup, "higher_is_better": False,
            "dtype": "f64 / f32", "data": "synthetic",
            "config": {"workload": "differentiation form: 8^3x16 x 8 DWF, eps=0.5, M5=1.8, mf=0.05, loss "
                                   "Re(eta^dag x), nvec=16, 4^4 blocks, Chebyshev filter order 100"},
            "c128": out["c128"], "c64": out["c64"]}


def _extents(spec: str) -> tuple:
    parts = [int(v) for v in spec.split(",")]
    return tuple(parts) if len(parts) == 4 else (parts[0],) * 4


def run_stencil(args, world, rank, local):
    """Repeated applications of H (Ls = 16) on random device data: the kernel-level
    workload the ncu captures in profiles/ run.  --lattice L or Lx,Ly,Lz,Lt;
    --dtype f64, f32 or h16 (FP16 storage); --reps launches timed after as many warm-up
    launches.  Reports the event-timed microseconds per launch and algorithmic GB/s."""
    import torch

    import paper_1611_06944_gb300 as hd
    torch.cuda.set_device(local)
    L, dtype, reps = _extents(args.lattice), args.dtype, args.reps
    h16 = dtype == "h16"
    dt = torch.complex64 if dtype in ("f32", "h16") else torch.complex128
    lat = hd.Lattice(L, LS)
    g = torch.Generator(device="cuda").manual_seed(0)
    U = torch.randn(4, lat.V4, 3, 3, dtype=dt, device="cuda", generator=g)
    x = torch.randn(args.nrhs, lat.V4, 12, LS, dtype=dt, device="cuda", generator=g)
    if h16:
        x = hd.encode_h16(lat, x)
    y = torch.empty_like(x)
    if args.variant >= 0:
        hd.stencil_tune(0, args.variant)
    apply = (lambda: hd.apply_g5dwf_h16(lat, U, x, M5, MF, out=y)) if h16 else \
        (lambda: hd.apply_g5dwf(lat, U, x, M5, MF, out=y))
    for _ in range(reps):
        apply()
    torch.cuda.synchronize()
    hd.stencil_timer(True)
    for _ in range(reps):
        apply()
    torch.cuda.synchronize()
    t = hd.stencil_timer_read("h16" if h16 else dt)
    hd.stencil_timer(False)
    chosen = hd.stencil_tune_info(lat, args.nrhs)["variant"] if dtype == "f32" and args.variant < 0 else args.variant
    us = t["ms"] / max(t["launches"], 1) * 1e3
    real = 4 if dt == torch.complex64 else 8
    per_site = 2 * 24 * real + 4 * 18 * real / LS / args.nrhs  # psi in + out, links shared by the Ls sites
    if h16:
        per_site = 2 * 52 + 4 * 18 * 4 / LS / args.nrhs        # half2 spinor + FP32 scale in and out; FP32 links
    gbs = lat.V5 * args.nrhs * per_site / (us * 1e-6) / 1e9
    return {"workload_kind": "stencil", "lattice": list(L), "Ls": LS, "dtype": dtype, "nrhs": args.nrhs,
            "us_per_launch": round(us, 2), "GBs": round(gbs, 1), "frac_of_hbm": round(gbs / peaks()["hbm_gbs"], 4),
            "bytes_per_site": per_site, "launches": t["launches"], "variant": chosen}


def run_coarse(args, world, rank, local):
    """Builds of the little Dirac operator from nvec random basis vectors on 4^4 blocks
    (Ls = 16): --lattice, --nvec, --dtype f64, f32 or f32fast (single-pass TF32
    projections), --reps timed builds after one warm-up; reported in units of one fine
    application of H of the same precision."""
    import torch

    import paper_1611_06944_gb300 as hd
    torch.cuda.set_device(local)
    L, nvec, dtype, reps = _extents(args.lattice), args.nvec, args.dtype, args.reps
    fast = dtype == "f32fast"
    dt = torch.complex64 if dtype in ("f32", "f32fast") else torch.complex128
    lat = hd.Lattice(L, LS)
    g = torch.Generator(device="cuda").manual_seed(0)
    U = torch.randn(4, lat.V4, 3, 3, dtype=torch.complex128, device="cuda", generator=g)
    v = torch.randn(nvec, lat.V4, 12, LS, dtype=torch.complex128, device="cuda", generator=g)
    sub = hd.subspace_from_vectors(lat, BLOCK, v, store_dtype=dt)
    del v
    torch.cuda.empty_cache()
    hd.build_coarse_op(sub, U, M5, MF, op_dtype=dt, fast=fast).close()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(reps):
        hd.build_coarse_op(sub, U, M5, MF, op_dtype=dt, fast=fast).close()
    e1.record()
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / reps
    Ud = U.to(dt)
    x = torch.randn(lat.V4, 12, LS, dtype=dt, device="cuda", generator=g)
    y = torch.empty_like(x)
    for _ in range(3):
        hd.apply_g5dwf(lat, Ud, x, M5, MF, out=y)
    torch.cuda.synchronize()
    e0.record()
    for _ in range(10):
        hd.apply_g5dwf(lat, Ud, x, M5, MF, out=y)
    e1.record()
    torch.cuda.synchronize()
    mv = e0.elapsed_time(e1) / 10
    sub.close()
    return {"workload_kind": "coarse", "lattice": list(L), "Ls": LS, "nvec": nvec, "block": list(BLOCK),
            "dtype": dtype, "build_ms": round(ms, 3), "fine_matvec_ms": round(mv, 4),
            "fine_matvecs": round(ms / mv, 1)}


def main(argv=None) -> int:
    ap = argparse.ArgumentParser(description=__doc__, formatter_class=argparse.RawDescriptionHelpFormatter)
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--workload", choices=["two-level", "precision", "batching", "table1", "differentiation",
                                           "stencil", "coarse"], default="two-level")
    ap.add_argument("--lattice", default="16", help="stencil/coarse: L or Lx,Ly,Lz,Lt (Ls = 16)")
    ap.add_argument("--dtype", default="f32", help="stencil: f64|f32|h16; coarse: f64|f32|f32fast")
    ap.add_argument("--nvec", type=int, default=24, help="coarse: basis vectors")
    ap.add_argument("--nrhs", type=int, default=1, help="stencil: fields per launch")
    ap.add_argument("--reps", type=int, default=4, help="stencil/coarse: timed launches or builds")
    ap.add_argument("--variant", type=int, default=-1,
                    help="stencil f32: run this tile variant (0-5 L1-tiled, 6 TMA-staged) instead of tuning")
    args = ap.parse_args(argv)
    world, rank, local = dist_setup()
    if args.impl == "reference":
        line = run_reference(args, world, rank)
    else:
        import __graft_entry__  # noqa: F401  (puts the repo on sys.path)
        if args.workload == "precision":
            line = run_precision(args, world, rank, local) if rank == 0 else None
        elif args.workload == "batching":
            line = run_batching(args, world, rank, local) if rank == 0 else None
        elif args.workload == "table1":
            line = run_table1(args, world, rank, local) if rank == 0 else None
        elif args.workload == "differentiation":
            line = run_differentiation(args, world, rank, local) if rank == 0 else None
        elif args.workload == "stencil":
            line = run_stencil(args, world, rank, local) if rank == 0 else None
        elif args.workload == "coarse":
            line = run_coarse(args, world, rank, local) if rank == 0 else None
        else:
            line = run_ours(args, world, rank, local)
    if rank == 0 and line is not None:
        print(json.dumps(line), flush=True)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
