#!/usr/bin/env python
"""Benchmark of the FFT-accelerated macromodel solve (Eq. final) on one GB300.

Workload (default): 16 x 16 lattice of boxes meshed 4 x 4 per face
(K = 576 unknowns per box), 32 cell types -- a PEC patch (side uniform in
[0.15, 0.45] lambda) on a 0.76 mm eps_r = 3, tan delta = 0.001 slab,
seeded type map -- one normal-incidence x-polarised plane wave at 10 GHz.  Every input is built on the product path: overlap
map (C++ setup), offset tables and macromodels (GPU tabulation and Schur
complement), excitation (GPU).

A step is one solve to relative residual 1e-6: flexible GMRES(30),
right-preconditioned by the near-field preconditioner (restricted additive
Schwarz by cells, one mesh layer of overlap), with the FP32 operator inside
FP64 residual refinement (MIXED).  The unpreconditioned MIXED and FP64
solves, the matvec rates, the CPU oracle and an end-to-end call with host
buffers are measured beside it.  One JSON line on rank 0.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]
"""
import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "solve time to 1e-6 residual & matvec GB/s vs FP64 plain; p50/p99 serve latency"
RTOL = 1e-6
RESTART = 30
# Products of the FP64-operator GMRES(30) solve of the default workload
# (16x16 patch-on-slab cells) to 1e-6 without a preconditioner: the oracle's
# GMRES is the same algorithm on the same operator, so it needs the same
# count; it is counted by the GPU solve (the bench line's fp64_plain.n_matvec)
# because the oracle, at ~1.8 s per product, would need over two hours.
REF_MATVECS_PER_SOLVE = 4129
FALLBACK_HBM_GBS = 6800.0
PC_OVERLAP = 1.0               # preconditioner margin, in mesh cells (a / n)
# DRAM bytes (read + write) per bin of one binmul_tma_kernel launch, from an
# ncu capture of the 12x12 lattice (576 bins, dram__bytes_read.sum +
# dram__bytes_write.sum); the kernel streams each bin's blocks once, so
# traffic scales with the bin count.
BINMUL_DRAM_BYTES_PER_BIN = (767108096 + 5353216) / 576
# the same for binmul_tma_pair_kernel (half spectrum) per stored bin, from
# the capture of the 12x12 lattice (290 stored bins)
PAIR_DRAM_BYTES_PER_STORED_BIN = (387588096 + 3930624) / 290
# binmul_orbit_kernel (one stored bin per mirror orbit of 8), from the capture
# of the 16x16 lattice itself (153 stored bins)
ORBIT_DRAM_BYTES_PER_STORED_BIN = (207879936 + 4441344) / 153


FALLBACK_BF16_TFLOPS = 1900.0


def peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return float(d.get("hbm_gbs", FALLBACK_HBM_GBS)), "measured"
    return FALLBACK_HBM_GBS, "fallback"


def bf16_peak():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        if "bf16_tflops" in d:
            return float(d["bf16_tflops"]), "measured"
    return FALLBACK_BF16_TFLOPS, "fallback"


MULTI_RHS = 32


def variant_section(B, W, torch, w, steps, **create_kw):
    """The same solve on a handle built with other options (create_kw of
    build_problem): time per solve, per bin multiply, per preconditioner
    apply and per FP32 product."""
    h, V, nu, _, _ = build_problem(B, W, torch, w, B.MIXED, **create_kw)
    X = torch.zeros_like(V)
    kw = dict(rtol=RTOL, restart=RESTART, max_iters=20000, max_refine=20, solver=B.SOLVER_MIXED)
    for _ in range(2):
        B.emsurf_solve(h, V, X, **kw)
    B.emsurf_profile_phases(h, ["binmul32", "precond"])
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(steps):
        st, info = B.emsurf_solve(h, V, X, **kw)
    e1.record()
    torch.cuda.synchronize()
    B.emsurf_profile(h, False)
    bin_ms, bin_n = B.emsurf_profile_read(h, "binmul32")
    pc_ms, pc_n = B.emsurf_profile_read(h, "precond")
    form, per = B.emsurf_operator_layout(h)
    out = {"options": {k: bool(v) for k, v in create_kw.items()},
           "spectrum": {0: "every bin", 1: "one bin per (k, -k) pair",
                        2: "one bin per mirror orbit of %d" % per}[form],
           "stored_bins": B.emsurf_operator_info(h)[0], "solve_ms": round(e0.elapsed_time(e1) / steps, 3),
           "converged": info[0]["converged"], "rel_residual": info[0]["rel_residual"],
           "iters": info[0]["iters"], "refinements": info[0]["refinements"],
           "binmul_ms_per_product": round(bin_ms / max(bin_n, 1), 5),
           "precond_ms_per_apply": round(pc_ms / max(pc_n, 1), 5),
           "fp32_matvec_ms": round(time_matvec(B, torch, h, nu, 1, B.FP32), 4)}
    h.close()
    torch.cuda.empty_cache()
    return out


def multi_rhs_section(B, W, torch, w, hbm):
    """FP32 products with MULTI_RHS right-hand sides: the tensor-core bin
    multiply (BF16x3) against the FP32 register-blocked kernel."""
    out = {"R": MULTI_RHS}
    tflops_peak, tkind = bf16_peak()
    for tc in (True, False):
        h, _, nu, _, _ = build_problem(B, W, torch, w, B.FP32, precond=False, max_rhs=MULTI_RHS,
                                    tensor_cores=tc)
        px, py, _ = B.emsurf_query(h)
        P = px * py
        x = torch.randn((MULTI_RHS, nu), dtype=torch.complex128, device="cuda")
        y = torch.empty_like(x)
        for _ in range(3):
            B.emsurf_matvec(h, x, y, B.FP32)
        torch.cuda.synchronize()
        B.emsurf_profile(h, True)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        reps = 10
        e0.record()
        for _ in range(reps):
            B.emsurf_matvec(h, x, y, B.FP32)
        e1.record()
        torch.cuda.synchronize()
        B.emsurf_profile(h, False)
        bm, n = B.emsurf_profile_read(h, "binmul32")
        bm /= max(n, 1)
        ph = {k: round(B.emsurf_profile_read(h, k)[0] / reps, 4) for k in ("fft32", "mm32", "scatter")}
        useful = 32.0 * w.E * w.E * MULTI_RHS * P        # complex MACs x 8 flops
        spec = 2 * w.E * w.E * P * 8                     # complex64 spectrum (= bf16 hi + lo)
        key = "tensor_bf16x3" if tc else "fp32_simt"
        out[key] = {"matvec_ms": round(e0.elapsed_time(e1) / reps, 3), "binmul_ms": round(bm, 4),
                    "useful_tflops": round(useful / bm / 1e9, 1),
                    "spectrum_gbs": round(spec / bm / 1e6, 1), "other_phases_ms": ph}
        if tc:
            # MMA work issued: 3 split passes x 2 operators x 2 M N K per bin, with
            # M = 128 per 32 rhs, N = 2E in chunks of 96, K = E in stages of 64
            groups, chunks, nk = -(-MULTI_RHS // 32), -(-2 * w.E // 96), -(-w.E // 64)
            executed = 3 * 2 * 2.0 * (128 * groups) * (96 * chunks) * (64 * nk) * P
            out[key]["tensor_tflops_executed"] = round(executed / bm / 1e9, 1)
            out[key]["tensor_frac"] = round(executed / bm / 1e9 / tflops_peak, 4)
            out[key]["hbm_frac"] = round(spec / bm / 1e6 / hbm, 4)
            out[key]["peak_kind"] = tkind
        h.close()
        torch.cuda.empty_cache()
    out["speedup"] = round(out["fp32_simt"]["binmul_ms"] / out["tensor_bf16x3"]["binmul_ms"], 2)
    return out


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled during the timed region."""
    FIELDS = ["clocks.sm", "clocks.max.sm", "clocks_event_reasons.hw_slowdown",
              "clocks_event_reasons.hw_thermal_slowdown", "clocks_event_reasons.sw_thermal_slowdown",
              "clocks_event_reasons.sw_power_cap"]

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), "--query-gpu=" + ",".join(self.FIELDS),
                 "--format=csv,noheader,nounits", "-lms", "100"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except OSError:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for l in self.lines:
            parts = [p.strip() for p in l.split(",")]
            if len(parts) != len(self.FIELDS):
                continue
            try:
                sm.append(float(parts[0]))
                smax.append(float(parts[1]))
            except ValueError:
                continue
            for n, v in zip(names, parts[2:]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(smax) if smax else None, "reasons": sorted(reasons),
                "samples": len(sm)}


def _rcs_grid(step_deg):
    th = np.radians(np.arange(0.0, 180.0 + 1e-9, step_deg))
    ph = np.radians(np.arange(0.0, 360.0, step_deg))
    TH, PH = np.meshgrid(th, ph, indexing="ij")
    return np.stack([np.sin(TH) * np.cos(PH), np.sin(TH) * np.sin(PH), np.cos(TH)], -1).reshape(-1, 3)


def _rcs(B, torch, h, w, zl, X, rhat):
    from paper_1911_04576_gb300 import workloads as W_
    F = torch.empty((X.shape[0], len(rhat), 3), dtype=torch.complex128, device="cuda")
    rcs = torch.empty((X.shape[0], len(rhat)), dtype=torch.float64, device="cuda")
    B.emsurf_far_field(h, W_.PERIOD, W_.PERIOD, W_.BOX_H, w.n, W_.K0, X, rhat, F, rcs, zlevels=zl)
    del F
    return rcs


def _db_diff(a, b, floor_db=40.0):
    """max |10 log10(a/b)| over directions where b > max(b) - floor_db (per rhs)."""
    a, b = np.asarray(a), np.asarray(b)
    out = 0.0
    for r in range(b.shape[0]):
        bd = 10 * np.log10(np.maximum(b[r], 1e-300))
        ad = 10 * np.log10(np.maximum(a[r], 1e-300))
        keep = bd > bd.max() - floor_db
        out = max(out, float(np.abs(ad[keep] - bd[keep]).max()))
    return out


def _timed(fn):
    import torch
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    r = fn()
    torch.cuda.synchronize()
    return r, (time.perf_counter() - t0) * 1e3


def _binmul_live(B, torch, h, x, prec, reps):
    """CUDA-event average of the bin multiply over `reps` products (the
    phase timer records on the product's stream) and the products' average."""
    y = torch.empty_like(x)
    B.emsurf_matvec(h, x, y, prec)
    B.emsurf_profile_phases(h, ["binmul32" if prec == B.FP32 else "binmul64"])
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record()
    for _ in range(reps):
        B.emsurf_matvec(h, x, y, prec)
    e1.record()
    torch.cuda.synchronize()
    B.emsurf_profile(h, False)
    ms, n = B.emsurf_profile_read(h, "binmul32" if prec == B.FP32 else "binmul64")
    return ms / max(n, 1), e0.elapsed_time(e1) / reps


def many_rhs_section(B, W, torch, name, hbm, bf16, time_left_s, rcs_step, max_iters=20000):
    """A many-right-hand-side configuration measured end to end on the
    product path: setup, FP32 (tensor-core) and FP64-accuracy products with
    all rhs, the preconditioner apply, the MIXED solve of all rhs to 1e-6,
    and the bistatic RCS of every rhs on a rcs_step-degree grid; the
    tensor-core bin multiply's live average against the HBM roofline."""
    w = W.WORKLOADS[name]
    t_start = time.time()
    h, V, nu, setup, zl = build_problem(B, W, torch, w, B.MIXED, max_rhs=w.n_rhs, tensor_cores=True)
    setup["total_s"] = round(time.time() - t_start, 2)
    _log(name + " setup", setup)
    px, py, dev_bytes = B.emsurf_query(h)
    P = px * py
    out = {"workload": w.name, "lattice": [w.nx, w.ny], "K": w.K, "n_types": w.n_types,
           "type_map": w.type_rule, "unknowns": nu, "rhs": w.n_rhs, "grid": [px, py],
           "setup": setup, "device_bytes": dev_bytes}
    x = torch.randn((w.n_rhs, nu), dtype=torch.complex128, device="cuda")
    bm32, mv32 = _binmul_live(B, torch, h, x, B.FP32, 5)
    kc, ns, tms = B.emsurf_tc_tuning(h)
    out["tc_autotune"] = {"picked": "%d sources x %d stages" % (kc, ns),
                          "ms_32x5": round(tms[0], 4), "ms_64x2": round(tms[1], 4)}
    spec = 2 * w.E * w.E * P * 8                       # bf16 hi + lo planes = complex64 bytes
    useful = 32.0 * w.E * w.E * w.n_rhs * P            # complex MACs x 8 flops
    out["fp32_matvec_ms"] = round(mv32, 3)
    out["roofline"] = {"kernel": "binmul_tc_kernel (bin multiply, BF16x3 on tcgen05, %d rhs)" % w.n_rhs,
                       "bound": "hbm", "achieved": round(spec / bm32 / 1e6, 1), "peak": hbm, "unit": "GB/s",
                       "frac": round(spec / bm32 / 1e6 / hbm, 4), "avg_launch_ms": round(bm32, 4),
                       "alg_bytes_per_launch": spec, "useful_tflops": round(useful / bm32 / 1e9, 1),
                       "useful_frac_of_bf16_peak": round(useful / bm32 / 1e9 / bf16, 4)}
    bm64, mv64 = _binmul_live(B, torch, h, x, B.FP64, 1)
    out["fp64_accuracy_matvec_ms"] = round(mv64, 2)
    out["fp64_accuracy_binmul+macromodel_ms"] = round(bm64, 2)
    r = torch.randn_like(V)
    y = torch.empty_like(V)
    B.emsurf_precond_apply(h, r, y)
    _, t = _timed(lambda: [B.emsurf_precond_apply(h, r, y) for _ in range(5)])
    out["precond_apply_ms"] = round(t / 5, 3)
    del x, r, y
    if time.time() - t_start > time_left_s:
        out["skipped"] = "time limit before the solve"
        h.close()
        return out
    X = torch.zeros_like(V)
    B.emsurf_profile(h, True)
    (st, info), t = _timed(lambda: B.emsurf_solve(h, V, X, rtol=RTOL, restart=RESTART, max_iters=max_iters,
                                                  max_refine=20, solver=B.SOLVER_MIXED))
    B.emsurf_profile(h, False)
    out["solve"] = {"rtol": RTOL, "max_iters": max_iters, "ms": round(t, 1), "status": st,
                    "ms_per_iter": round(t / max(1, info[0]["iters"]), 3), "iters": info[0]["iters"],
                    "refinements": info[0]["refinements"], "n_matvec": info[0]["n_matvec"],
                    "all_converged": all(i["converged"] for i in info),
                    "max_rel_residual": max(i["rel_residual"] for i in info),
                    "phases_ms": {p: round(B.emsurf_profile_read(h, p)[0], 1) for p in B.PHASES}}
    if time.time() - t_start < time_left_s:
        rhat = _rcs_grid(rcs_step)
        rcs, t = _timed(lambda: _rcs(B, torch, h, w, zl, X, rhat))
        s = rcs.cpu().numpy()
        out["rcs"] = {"grid_deg": rcs_step, "directions": len(rhat), "rhs": w.n_rhs, "ms": round(t, 1),
                      "max_dbsm": round(float(10 * np.log10(s.max())), 2)}
    B.emsurf_check(h)
    h.close()
    out["total_s"] = round(time.time() - t_start, 1)
    return out


def accuracy_section(B, torch, h, V, X_bench, w, zl):
    """Result-level accuracy of the MIXED path against the FP64-operator
    GMRES solved to 1e-11 (both preconditioned): currents (rel-L2) and
    bistatic RCS (dB, where sigma > sigma_max - 40 dB) on a 2-degree grid,
    for the bench's rtol and for the configuration's rtol 1e-8."""
    X64 = torch.zeros_like(V)
    (st, info64), t64 = _timed(lambda: B.emsurf_solve(h, V, X64, rtol=1e-11, restart=RESTART, max_iters=20000,
                                                      solver=B.SOLVER_FP64))
    X8 = torch.zeros_like(V)
    (st8, info8), t8 = _timed(lambda: B.emsurf_solve(h, V, X8, rtol=1e-8, restart=RESTART, max_iters=20000,
                                                     max_refine=20, solver=B.SOLVER_MIXED))
    X8f = torch.zeros_like(V)
    (st8f, info8f), t8f = _timed(lambda: B.emsurf_solve(h, V, X8f, rtol=1e-8, restart=RESTART, max_iters=20000,
                                                        solver=B.SOLVER_FP64))
    rhat = _rcs_grid(2.0)
    s64 = _rcs(B, torch, h, w, zl, X64, rhat).cpu().numpy()
    out = {"reference": "FP64-operator GMRES(30) + preconditioner to rtol 1e-11 (%d iters, %.1f ms)"
                        % (info64[0]["iters"], t64),
           "rcs_grid": "2 deg, %d directions; dB compared where sigma > sigma_max - 40 dB" % len(rhat)}
    for key, X, t, info in (("mixed_rtol_1e-6", X_bench, None, None), ("mixed_rtol_1e-8", X8, t8, info8)):
        xm = X.cpu().numpy()
        x64 = X64.cpu().numpy()
        sm = _rcs(B, torch, h, w, zl, X, rhat).cpu().numpy()
        out[key] = {"currents_rel_l2": float(np.linalg.norm(xm - x64) / np.linalg.norm(x64)),
                    "rcs_max_db": round(_db_diff(sm, s64), 5)}
        if t is not None:
            out[key]["solve_ms"] = round(t, 2)
            out[key]["iters"] = info[0]["iters"]
    out["fp64_rtol_1e-8"] = {"solve_ms": round(t8f, 2), "iters": info8f[0]["iters"],
                             "converged": info8f[0]["converged"]}
    return out


def cpu_fft_section(W, w, nmv_plain, iters_pc):
    """The timed CPU FFT baseline (complex128, scipy.fft with every host core
    plus batched per-bin products): spectrum build, products, and GMRES
    iterations with that product; the solve time is extrapolated by the
    GPU FP64 GMRES(30)'s product count on the same operator."""
    from oracle import cpu_fft, lattice, solve
    from oracle.mesh import box_mesh
    A = W.PERIOD
    idx, sgn, nu = lattice.overlap_map(box_mesh(A, A, W.BOX_H, w.n), w.nx, w.ny, A, A)
    Lt, Kt = W.random_tables(w.nx, w.ny, w.E, 1)
    Z = W.random_macromodels(w.n_types, w.K, 2)
    coef = (1j * W.K0, 1.0, -1.0, 1j * W.K0)
    px, py = 2 * w.nx, 2 * w.ny
    t0 = time.perf_counter()
    Lh, Kh = cpu_fft.spectrum(Lt, Kt, px, py)
    t_spec = time.perf_counter() - t0
    del Lt, Kt
    tm = W.type_map(w)
    x = W.random_vectors(1, nu, 3)[0]
    mv = lambda v: cpu_fft.matvec(v, Lh, Kh, coef, Z, tm, idx, sgn, nu, w.nx, w.ny)
    mv(x)
    t0 = time.perf_counter()
    for _ in range(3):
        mv(x)
    t_mv = (time.perf_counter() - t0) / 3
    t0 = time.perf_counter()
    _, it, _ = solve.gmres(mv, x, rtol=1e-30, restart=RESTART, max_iters=6)
    t_it = (time.perf_counter() - t0) / max(it, 1)
    return {"kind": "CPU FFT product (complex128, scipy.fft + batched per-bin matmul)",
            "cores": len(os.sched_getaffinity(0)), "grid": [px, py], "spectrum_s": round(t_spec, 2),
            "matvec_ms": round(t_mv * 1e3, 1), "gmres_iter_ms": round(t_it * 1e3, 1),
            "fp64_plain_solve_ms_extrapolated": round(t_it * 1e3 * nmv_plain, 0),
            "note": "solve = GMRES(30) iteration time x the %d products of the GPU FP64 solve (same "
                    "operator, same algorithm); unpreconditioned (the GPU preconditioned solve takes %d "
                    "iterations)" % (nmv_plain, iters_pc)}


_T0 = time.time()


def _log(section, obj=None):
    """Progress on stderr: seconds since start, the section, its result (so a
    run cut short still shows where the time went and what was measured)."""
    print("[bench %7.1fs] %s %s" % (time.time() - _T0, section, json.dumps(obj) if obj is not None else ""),
          file=sys.stderr, flush=True)


def last_iters(infos):
    return infos[-1]["iters"] if infos else 0


def max_over_ranks(dist, value, device):
    """The largest of every rank's value (a job takes as long as its slowest
    rank); value itself without a process group."""
    if dist is None:
        return value
    import torch
    t = torch.tensor([float(value)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return t.item()


def dist_init():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def build_problem(B, W, torch, w, precision, precond=True, max_rhs=None, tensor_cores=False, mirrors=False,
                  precond_int8=False):
    """Product-path setup (untimed): U_o, tables, macromodels, handle with
    the near-field preconditioner, V."""
    A, H = W.PERIOD, W.BOX_H
    coef = (1j * W.K0, 1.0, -1.0, 1j * W.K0)
    idx, sgn, nu = B.emsurf_setup_overlap(w.n, w.nx, w.ny)
    xy = B.emsurf_setup_unknown_xy(A, A, H, w.n, w.nx, w.ny, idx, nu) if precond else None
    zl = B.emsurf_setup_slab_zlevels(H, w.n, W.SLAB_T)     # box rows end at the slab top
    L = torch.empty((2 * w.ny - 1, 2 * w.nx - 1, w.E, w.E), dtype=torch.complex128, device="cuda")
    K = torch.empty_like(L)
    t0 = time.time()
    B.emsurf_tabulate_offsets(A, A, H, w.n, w.nx, w.ny, W.K0, L, K, zlevels=zl)
    t_tab = time.time() - t0
    Z = torch.empty((w.n_types, w.K, w.K), dtype=torch.complex128, device="cuda")
    t0 = time.time()
    B.emsurf_macromodel_slab_patch(A, A, H, w.n, zl, W.patch_sides(w), w.patch_n, W.RING_LAYERS,
                                   W.EPS_SLAB, W.K0, Z)
    torch.cuda.synchronize()
    t_mm = time.time() - t0
    t0 = time.time()
    h = B.emsurf_create(w.nx, w.ny, w.E, nu, W.type_map(w), Z, L, K, coef, idx, sgn,
                        precision=precision, max_rhs=max_rhs or w.n_rhs, tables_on_device=True,
                        unknown_xy=xy, cell=(A, A),
                        precond_overlap=PC_OVERLAP * A / w.n if precond else 0.0,
                        tensor_cores=tensor_cores,
                        mirrors=B.emsurf_setup_box_mirrors(A, A, w.n) if mirrors else None,
                        precond_int8=precond_int8)
    torch.cuda.synchronize()
    t_create = time.time() - t0
    del L, K, Z
    torch.cuda.empty_cache()
    waves = W.plane_waves(w)
    V = torch.empty((w.n_rhs, nu), dtype=torch.complex128, device="cuda")
    B.emsurf_excitation(h, A, A, H, w.n, W.K0, np.array([k for k, _ in waves]),
                        np.array([e for _, e in waves]), V, zlevels=zl)
    return h, V, nu, {"tabulate_s": round(t_tab, 3), "macromodels_s": round(t_mm, 3),
                      "create_s": round(t_create, 3)}, zl


def time_matvec(B, torch, h, nu, R, prec, reps=10):
    x = torch.randn((R, nu), dtype=torch.complex128, device="cuda")
    y = torch.empty_like(x)
    for _ in range(3):
        B.emsurf_matvec(h, x, y, prec)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record()
    for _ in range(reps):
        B.emsurf_matvec(h, x, y, prec)
    e1.record()
    torch.cuda.synchronize()
    return e0.elapsed_time(e1) / reps


def cpu_oracle_matvec_seconds(W, w, nu_expected):
    """One full FFT-free oracle product (Eq. MVP by the direct offset sum) on
    random tables of the workload's shapes -- values do not change its cost."""
    from oracle import lattice
    from oracle.mesh import box_mesh
    A = W.PERIOD
    idx, sgn, nu = lattice.overlap_map(box_mesh(A, A, W.BOX_H, w.n), w.nx, w.ny, A, A)
    assert nu == nu_expected
    Lt, Kt = W.random_tables(w.nx, w.ny, w.E, 1)
    Z = W.random_macromodels(w.n_types, w.K, 2)
    x = W.random_vectors(1, nu, 3)[0]
    t0 = time.perf_counter()
    lattice.matvec_direct(x, Lt, Kt, (1j * W.K0, 1.0, -1.0, 1j * W.K0), Z, W.type_map(w), idx, sgn,
                          nu, w.nx, w.ny)
    return time.perf_counter() - t0


SERVE_SIZES = (8, 16, 24, 32, 64)   # lattice N x N of the serving stream
SERVE_MESH = (3, 4)            # boxes meshed n x n: K = 324 or 576
SERVE_RHS = tuple(range(1, 17))   # rhs per request, uniform in 1..16
SERVE_RATE = 1.0               # Poisson arrivals per second (default; --serve-rate)
SERVE_MAX_MS = 20000.0         # wall-time limit of each request's solve
SERVE_DRAIN_S = 20.0           # after the last arrival: queued requests are withdrawn
SERVE_BUDGET = 80 << 30        # device-memory budget of the server
SERVE_FP64_SAMPLE = 4         # requests of the one-at-a-time FP64 arm
SERVE_FP64_WINDOW_S = 30.0     # and its window (later requests are withdrawn)


def serve_requests(B, W, nreq, seed, precision, precond, rate=SERVE_RATE):
    """The seeded stream: Poisson arrival times and the requests (lattice,
    mesh, rhs, type map, plane waves) drawn as the serving configuration
    says, cells from one 32-type patch-on-slab library."""
    rng = np.random.default_rng(seed)
    lib_sides = rng.uniform(0.15, 0.45, 32) * W.LAMBDA
    arrivals = np.cumsum(rng.exponential(1.0 / rate, nreq))
    reqs = []
    for _ in range(nreq):
        N = int(rng.choice(SERVE_SIZES))
        n = int(rng.choice(SERVE_MESH))
        R = int(rng.choice(SERVE_RHS))
        th = rng.uniform(0.0, 60.0, R)
        ph = rng.choice([0.0, 90.0], R)
        waves = [W.plane_waves(W.Workload("s", 1, 1, 1, 1, 0, 0, angles=[(t, p, "theta")]))[0]
                 for t, p in zip(th, ph)]
        reqs.append(dict(a=W.PERIOD, b=W.PERIOD, h=W.BOX_H, n=n, nx=N, ny=N, k0=W.K0,
                         patch_sides=lib_sides, patch_z=W.PATCH_Z, patch_n=4,
                         type_map=rng.integers(0, 32, N * N), khat=np.array([w_[0] for w_ in waves]),
                         ehat=np.array([w_[1] for w_ in waves]), precision=precision, rtol=RTOL,
                         restart=RESTART, max_iters=20000, max_refine=20, max_ms=SERVE_MAX_MS,
                         precond_overlap=PC_OVERLAP * W.PERIOD / n if precond else 0.0,
                         slab_t=W.SLAB_T, slab_eps=W.EPS_SLAB, ring_layers=W.RING_LAYERS))
    return arrivals, reqs


_ABANDONED = []     # servers left with a request that did not end (kept alive, never destroyed)


def serve_stream(B, W, arrivals, reqs, max_active, cache, window_s):
    """Submit the requests at their arrival times (those arriving within
    window_s); when the window closes, withdraw the ones still queued and
    collect the running ones (each solve is bounded by its max_ms).
    Latency percentiles over the completed requests, throughput over the
    makespan."""
    sv = B.emsurf_server_create(0, SERVE_BUDGET, max_active, cache=cache)
    pending, res, refused, offered = [], [], 0, 0
    described = {}

    def collect():
        keep = []
        for t in pending:
            r = B.emsurf_poll(sv, t)
            if r is None:
                keep.append(t)
            else:
                res.append(r)
        return keep
    t0 = time.perf_counter()
    for at, r in zip(arrivals, reqs):
        if at > window_s:
            break
        dt = t0 + at - time.perf_counter()
        if dt > 0:
            time.sleep(dt)
        offered += 1
        q, keep = B.make_request(**r)
        try:
            t = B.emsurf_submit(sv, q, keep)
            pending.append(t)
            described[t] = {"nx": r["nx"], "n": r["n"], "rhs": len(r["khat"]), "arrival_s": round(float(at), 2)}
        except B.EmsurfError as e:
            if e.status != B.EMSURF_EBUSY:
                raise
            refused += 1
        pending = collect()
    while pending and time.perf_counter() - t0 < window_s:
        time.sleep(0.05)
        pending = collect()
    withdrawn = sum(1 for t in pending if B.emsurf_cancel(sv, t))
    _log("serve window closed", {"completed": len(res), "withdrawn": withdrawn, "running": len(pending) - withdrawn})
    # the running requests: their solves end within max_ms; a request that
    # has not ended well after that is reported and left behind (the server
    # is then not destroyed, which would wait for it)
    unfinished = []
    for t in pending:
        try:
            r = B.emsurf_wait(sv, t, int(SERVE_MAX_MS + 180000))
        except B.EmsurfError as e:
            if e.status != B.EMSURF_ETIMEDOUT:
                raise
            d = dict(described.get(t) or {})
            d["phase"] = B.emsurf_request_phase(sv, t)
            unfinished.append(d)
            continue
        if r["status"] != B.EMSURF_ECANCELED:
            res.append(r)
    makespan = time.perf_counter() - t0
    stats = B.emsurf_server_stats(sv)
    if unfinished:
        _log("serve: requests still running at the end", unfinished)
        _ABANDONED.append(sv)
    else:
        sv.close()
    lat = np.array([r["latency_ms"] for r in res]) if res else np.zeros(1)
    mean = lambda k: round(float(np.mean([r[k] for r in res])), 1) if res else None
    offered_span = float(arrivals[offered - 1]) if offered else 0.0
    return {"offered": offered, "offered_rps": round(offered / max(offered_span, 1e-9), 2),
            "completed": len(res), "refused_ebusy": refused, "withdrawn_at_window_end": withdrawn,
            "converged": int(sum(r["status"] == B.EMSURF_OK for r in res)),
            "stopped_at_max_ms": int(sum(r["status"] == B.EMSURF_ENOTCONV for r in res)),
            "throughput_rps": round(len(res) / makespan, 3), "makespan_s": round(makespan, 2),
            "window_s": window_s,
            "p50_ms": round(float(np.percentile(lat, 50)), 1), "p99_ms": round(float(np.percentile(lat, 99)), 1),
            "mean_ms": round(float(lat.mean()), 1), "queue_ms_mean": mean("queue_ms"),
            "setup_ms_mean": mean("setup_ms"), "solve_ms_mean": mean("solve_ms"),
            "cache_hits": int(sum(r["cache_hit"] for r in res)),
            "cache": {"bytes": stats[0], "operators": stats[1], "libraries": stats[2], "evictions": stats[3]},
            "max_active": max_active, "unfinished": unfinished}


def serve_section(B, W, nreq, rate):
    arrivals, reqs = serve_requests(B, W, nreq, 7, B.MIXED, True, rate)
    window = float(arrivals[-1]) + SERVE_DRAIN_S
    out = {"stream": "Poisson %.2f/s, %d requests; lattices %s, K %s, rhs %d..%d, 32-type patch-on-slab "
                     "library; rtol %g; each solve limited to %.0f s; budget %d GB; near-field "
                     "preconditioner; MIXED requests with >= 8 rhs use the tensor-core bin multiply; "
                     "requests still queued %.0f s after the last arrival are withdrawn"
                     % (rate, nreq, list(SERVE_SIZES), [36 * m * m for m in SERVE_MESH], SERVE_RHS[0],
                        SERVE_RHS[-1], RTOL, SERVE_MAX_MS / 1e3, SERVE_BUDGET >> 30, SERVE_DRAIN_S),
           "mixed_batched_resident": serve_stream(B, W, arrivals, reqs, 4, True, window)}
    _log("serve mixed arm", out["mixed_batched_resident"])
    # the FP64 reference arm, one request at a time and nothing kept between
    # requests, on the first requests of the same stream (a bounded sample)
    k = min(SERVE_FP64_SAMPLE, nreq)
    a64, r64 = serve_requests(B, W, nreq, 7, B.FP64, True, rate)
    out["fp64_one_at_a_time"] = serve_stream(B, W, a64[:k], r64[:k], 1, False, SERVE_FP64_WINDOW_S)
    out["fp64_one_at_a_time"]["sample"] = "first %d requests of the stream" % k
    return out


def reference_arm(args, W, w):
    ws, rank, _ = dist_init()
    if rank != 0:
        return
    from oracle import lattice
    from oracle.mesh import box_mesh
    A = W.PERIOD
    idx, sgn, nu = lattice.overlap_map(box_mesh(A, A, W.BOX_H, w.n), w.nx, w.ny, A, A)
    Lt, Kt = W.random_tables(w.nx, w.ny, w.E, 1)
    Z = W.random_macromodels(w.n_types, w.K, 2)
    coef = (1j * W.K0, 1.0, -1.0, 1j * W.K0)
    x = W.random_vectors(1, nu, 3)[0]
    tm = W.type_map(w)
    nmv = REF_MATVECS_PER_SOLVE
    times = []
    for i in range(args.warmup + args.steps):
        t0 = time.perf_counter()
        lattice.matvec_direct(x, Lt, Kt, coef, Z, tm, idx, sgn, nu, w.nx, w.ny)
        dt = time.perf_counter() - t0
        if i >= args.warmup:
            times.append(dt)
    t_mv = statistics.mean(times)
    value = t_mv * 1e3 * nmv if nmv else None
    cores = len(os.sched_getaffinity(0))
    sample = ("one full oracle direct-offset product (Eq. MVP, no FFT) per step on the %s "
              "workload; solve time = per-product time x %s FP64 GMRES(30) products"
              % (w.name, nmv))
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": value, "unit": "ms", "n_gpus": ws,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": t_mv * 1e3,
        "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic", "config": {"workload": w.name, "nx": w.nx, "ny": w.ny, "K": w.K,
                                        "unknowns": nu, "rtol": RTOL},
        "cpu_baseline": {"value": value, "unit": "ms", "cores": cores, "kind": "oracle",
                         "sample": sample, "matvec_s": t_mv},
        "e2e": {"value": value, "unit": "ms", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="lattice16x16_k576")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--multi-rhs", type=int, default=1,
                    help="also time %d-rhs FP32 products, tensor cores vs FP32 kernels (0 = skip)" % 32)
    ap.add_argument("--serve-requests", type=int, default=24,
                    help="requests of the serving stream (0 = skip the serving measurement)")
    ap.add_argument("--precond-int8", type=int, default=1,
                    help="also time the solve with 8-bit preconditioner rows (0 = skip)")
    ap.add_argument("--mirror-orbits", type=int, default=1,
                    help="also time the solve on a handle with one FP32 bin per mirror orbit (0 = skip)")
    ap.add_argument("--serve-rate", type=float, default=SERVE_RATE,
                    help="Poisson arrival rate of the serving stream (requests per second)")
    ap.add_argument("--matvecs-only", type=int, default=0,
                    help="profiler driver: build the workload, run this many products, exit")
    ap.add_argument("--precision", default="mixed", choices=["mixed", "fp32", "fp64"],
                    help="operators kept resident (--matvecs-only)")
    ap.add_argument("--rhs", type=int, default=0,
                    help="profiler driver: right-hand sides of the --matvecs-only products")
    ap.add_argument("--mirrors", type=int, default=0,
                    help="profiler driver: give the handle the box's mirrors (--matvecs-only)")
    ap.add_argument("--tensor-cores", action="store_true",
                    help="profiler driver: build the tensor-core planes (--matvecs-only)")
    ap.add_argument("--batched", type=int, default=1,
                    help="also measure the 48x48 / K = 576 / 32-plane-wave configuration (0 = skip)")
    ap.add_argument("--largest", type=int, default=1,
                    help="also measure the 100x100 / K = 324 / 8-plane-wave configuration (0 = skip)")
    ap.add_argument("--largest-iters", type=int, default=600,
                    help="GMRES iterations allowed to the 100x100 solve (0 = to convergence)")
    ap.add_argument("--accuracy", type=int, default=1,
                    help="also compare MIXED currents and RCS with an FP64 solve to 1e-11 (0 = skip)")
    ap.add_argument("--solve-iters", type=int, default=0,
                    help="profiler driver: with --matvecs-only, also run one mixed solve capped "
                         "at this many GMRES iterations")
    args = ap.parse_args()
    from paper_1911_04576_gb300 import workloads as W
    w = W.WORKLOADS[args.workload]
    if args.impl == "reference":
        reference_arm(args, W, w)
        return
    import torch
    from paper_1911_04576_gb300 import binding as B
    ws, rank, local = dist_init()
    torch.cuda.set_device(local)
    dist = None
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    cpu = None
    if args.matvecs_only:
        prec = {"mixed": B.MIXED, "fp32": B.FP32, "fp64": B.FP64}[args.precision]
        R = args.rhs or w.n_rhs
        h, V, nu, _, _ = build_problem(B, W, torch, w, prec, max_rhs=max(R, w.n_rhs),
                                    tensor_cores=args.tensor_cores, mirrors=bool(args.mirrors))
        for p in ((B.FP32,) if prec == B.FP32 else (B.FP64,) if prec == B.FP64 else (B.FP32, B.FP64)):
            x = torch.randn((R, nu), dtype=torch.complex128, device="cuda")
            y = torch.empty_like(x)
            for _ in range(args.matvecs_only):
                B.emsurf_matvec(h, x, y, p)
        if args.solve_iters and prec == B.MIXED:
            X = torch.zeros_like(V)
            B.emsurf_solve(h, V, X, rtol=RTOL, restart=RESTART, max_iters=args.solve_iters,
                           max_refine=20, solver=B.SOLVER_MIXED)
        torch.cuda.synchronize()
        h.close()
        return
    h, V, nu, setup, zl = build_problem(B, W, torch, w, B.MIXED)
    _log("setup", setup)
    X = torch.zeros_like(V)
    hbm, peak_kind = peaks()
    # FP64-plain reference solve on the same handle (FP64 operator GMRES,
    # no preconditioner), and the unpreconditioned MIXED solve
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    st64, info64 = B.emsurf_solve(h, V, X, rtol=RTOL, restart=RESTART, max_iters=20000,
                                  solver=B.SOLVER_FP64, precond=-1)
    t64 = (time.perf_counter() - t0) * 1e3
    t0 = time.perf_counter()
    stnp, infonp = B.emsurf_solve(h, V, X, rtol=RTOL, restart=RESTART, max_iters=20000,
                                  max_refine=20, solver=B.SOLVER_MIXED, precond=-1)
    tnp = (time.perf_counter() - t0) * 1e3
    t0 = time.perf_counter()
    st64p, info64p = B.emsurf_solve(h, V, X, rtol=RTOL, restart=RESTART, max_iters=20000,
                                    solver=B.SOLVER_FP64)
    t64p = (time.perf_counter() - t0) * 1e3
    pc_elems, pc_subtot, pc_nmax = B.emsurf_precond_info(h)
    _log("reference solves", {"fp64_plain_ms": t64, "mixed_unpreconditioned_ms": tnp, "fp64_precond_ms": t64p})
    # matvec rates
    R = w.n_rhs
    mv32 = time_matvec(B, torch, h, nu, R, B.FP32)
    mv64 = time_matvec(B, torch, h, nu, R, B.FP64)
    px, py, dev_bytes = B.emsurf_query(h)
    P = px * py
    stored, _ = B.emsurf_operator_info(h)        # FP32 spectrum bins held
    form, per_stored = B.emsurf_operator_layout(h)  # 0 full, 1 (k, -k) pairs, 2 mirror orbits
    bytes32 = 2 * w.E * w.E * stored * 8 + w.n_types * w.K * w.K * 8 + 2 * R * nu * 16
    # digit planes: 7 bytes per real number, sources in blocks of 16, read once per 6 rhs
    up16 = lambda m: -(-m // 16) * 16
    bytes64 = (-(-R // 6) * 2 * w.E * up16(w.E) * P + w.n_types * w.K * up16(w.K)) * 14 + 2 * R * nu * 16
    solve_kw = dict(rtol=RTOL, restart=RESTART, max_iters=20000, max_refine=20,
                    solver=B.SOLVER_MIXED)
    for _ in range(args.warmup):
        B.emsurf_solve(h, V, X, **solve_kw)
    # ------------------------------------------------------------ timed region
    clocks = ClockSampler(local)
    clocks.start()
    # only the dominant kernel is timed live (two events per product): the
    # full phase breakdown comes from a separate profiled solve below
    B.emsurf_profile_phases(h, ["binmul32"])
    launches0 = B.emsurf_launch_count(h)
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    infos = []
    for _ in range(args.steps):
        st, info = B.emsurf_solve(h, V, X, **solve_kw)
        infos.append(info[0])
    e1.record()
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    ms_total = e0.elapsed_time(e1)
    launches = B.emsurf_launch_count(h) - launches0
    B.emsurf_profile(h, False)
    clk = clocks.stop()
    bin_ms, bin_n = B.emsurf_profile_read(h, "binmul32")
    bin_ms_timed, bin_n_timed = bin_ms, bin_n
    # phase breakdown: one more solve (outside the timed region) with every
    # phase recorded; per-solve figures below are from this run
    B.emsurf_profile(h, True)
    B.emsurf_solve(h, V, X, **solve_kw)
    torch.cuda.synchronize()
    B.emsurf_profile(h, False)
    bin_ms, bin_n = B.emsurf_profile_read(h, "binmul32")
    mm_ms, mm_n = B.emsurf_profile_read(h, "mm32")
    fft_ms, fft_n = B.emsurf_profile_read(h, "fft32")
    bin64_ms, bin64_n = B.emsurf_profile_read(h, "binmul64")
    arn_ms, _ = B.emsurf_profile_read(h, "arnoldi")
    sct_ms, _ = B.emsurf_profile_read(h, "scatter")
    pc_ms, pc_n = B.emsurf_profile_read(h, "precond")
    fft64_ms, _ = B.emsurf_profile_read(h, "fft64")
    mm64_ms, _ = B.emsurf_profile_read(h, "mm64")
    ms = max_over_ranks(dist, ms_total / args.steps, "cuda")
    _log("timed solves", {"ms_per_solve": ms, "iters": infos[-1]["iters"] if infos else None})
    # ------------------------------------------------------------ end to end
    Vh = V.cpu().pin_memory()
    Xh = torch.empty_like(Vh).pin_memory()
    Vd = torch.empty_like(V)
    Xd = torch.empty_like(V)
    torch.cuda.synchronize()
    f0, f1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    f0.record()
    for _ in range(args.steps):
        Vd.copy_(Vh, non_blocking=True)
        B.emsurf_solve(h, Vd, Xd, **solve_kw)
        Xh.copy_(Xd, non_blocking=True)
    f1.record()
    torch.cuda.synchronize()
    e2e_ms = f0.elapsed_time(f1) / args.steps
    # ------------------------------------------------------------ accuracy
    accuracy = accuracy_section(B, torch, h, V, X, w, zl) if args.accuracy else None
    _log("accuracy", accuracy)
    # ------------------------------------------------------------ mirror orbits
    orbits = variant_section(B, W, torch, w, min(args.steps, 10), mirrors=True) if args.mirror_orbits else None
    _log("mirror_orbits", orbits)
    pc8 = variant_section(B, W, torch, w, min(args.steps, 10), precond_int8=True) if args.precond_int8 else None
    _log("precond_int8", pc8)
    # ------------------------------------------------------------ many rhs
    multi = multi_rhs_section(B, W, torch, w, hbm) if args.multi_rhs else None
    _log("multi_rhs", multi)
    h.close()          # free the bench handle's device memory for the other sections
    torch.cuda.empty_cache()
    bf16, _ = bf16_peak()
    batched = many_rhs_section(B, W, torch, "lattice48x48_k576_r32", hbm, bf16, 120.0, 1.0) \
        if args.batched else None
    _log("batched", batched)
    torch.cuda.empty_cache()
    # the largest array's solve is capped in the default run (its full solve
    # to 1e-6 takes ~4800 iterations); --largest-iters 0 lifts the cap
    largest = many_rhs_section(B, W, torch, "lattice100x100_k324_r8", hbm, bf16, 150.0, 2.0,
                               max_iters=args.largest_iters or 40000) if args.largest else None
    _log("largest", largest)
    torch.cuda.empty_cache()
    # ------------------------------------------------------------ serving
    serve = None
    if args.serve_requests > 0:
        _log("serve start")
        serve = serve_section(B, W, args.serve_requests, args.serve_rate)
        _log("serve", serve)
    # ------------------------------------------------------------ CPU oracle
    cpu_fft = None
    if rank == 0 and ws == 1 and not args.no_cpu_baseline:
        _log("cpu baselines start")
        cpu_fft = cpu_fft_section(W, w, info64[0]["n_matvec"], last_iters(infos))
        _log("cpu_fft", cpu_fft)
        t_cpu = cpu_oracle_matvec_seconds(W, w, nu)
        _log("cpu oracle product", {"s": round(t_cpu, 3)})
        nmv64 = info64[0]["n_matvec"]
        cpu = {"value": t_cpu * 1e3 * nmv64, "unit": "ms", "cores": len(os.sched_getaffinity(0)),
               "kind": "oracle",
               "sample": "one full oracle direct-offset product (Eq. MVP, FFT-free, complex128) "
                         "on the same workload shapes, %.2f s; solve = that x %d products of "
                         "the FP64 GMRES(30) solve" % (t_cpu, nmv64),
               "matvec_s": round(t_cpu, 3)}
    if rank != 0:
        if dist:
            dist.destroy_process_group()
        return
    bin_avg = bin_ms_timed / max(bin_n_timed, 1)     # live over the timed region
    # algorithmic bytes of the kernel that ran: the stored spectrum bins once,
    # X^ read and Y^ written for every bin
    alg_bin = 2 * w.E * w.E * stored * 8 + 2 * R * w.K * P * 8
    achieved = alg_bin / (bin_avg * 1e-3) / 1e9
    per_unit = {0: BINMUL_DRAM_BYTES_PER_BIN, 1: PAIR_DRAM_BYTES_PER_STORED_BIN,
                2: ORBIT_DRAM_BYTES_PER_STORED_BIN}[form]
    traffic = per_unit * (stored if form else P) if per_unit else None
    bin_kernel = {0: "binmul_tma_kernel (bin multiply, FP32)",
                  1: "binmul_tma_pair_kernel (bin multiply, FP32, half spectrum: %d of %d bins)" % (stored, P),
                  2: "binmul_orbit_kernel (bin multiply, FP32, one bin per mirror orbit of %d: %d of %d bins)"
                     % (per_stored, stored, P)}[form]
    # preconditioner apply: FP16 owned inverse rows (4 bytes per entry, one FP32
    # scale per row) once, r gathered, owned rows written
    pc_avg = pc_ms / max(pc_n, 1)
    alg_pc = pc_elems * 4 + nu * 4 + R * (pc_subtot * 16 + pc_subtot * 8 + nu * 16)
    pc_achieved = alg_pc / (pc_avg * 1e-3) / 1e9 if pc_n else None
    last = infos[-1]
    out = {
        "metric": METRIC, "value": round(ms, 3), "unit": "ms", "n_gpus": ws, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": round(ms, 3), "higher_is_better": False,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32+f64", "data": "synthetic",
        "config": {"workload": w.name, "nx": w.nx, "ny": w.ny, "K": w.K, "n_types": w.n_types,
                   "nrhs": R, "unknowns": nu, "grid": [px, py], "rtol": RTOL, "restart": RESTART,
                   "solver": "flexible GMRES(30), near-field RAS preconditioner (overlap %.1f "
                             "mesh cells), FP32 operator inside FP64 residual refinement"
                             % PC_OVERLAP,
                   "l2": "inputs larger than L2: %.2f GB complex64 + %.2f GB complex128 "
                         "Fourier-domain blocks" % (bytes32 / 1e9, bytes64 / 1e9),
                   "parallelism": "replicas" if ws > 1 else "single"},
        "solve": {"iters": last["iters"], "refinements": last["refinements"],
                  "n_matvec": last["n_matvec"], "rel_residual": last["rel_residual"],
                  "converged": last["converged"]},
        "operator_arithmetic": {"fp32": "complex64 operator, FP32 arithmetic (inner GMRES)",
                                "fp64_accuracy": "FP64-operator products from exact base-256 digits "
                                                 "of 55-bit integers on the tensor cores (FP64 "
                                                 "accuracy); FP64 FFTs, residuals, orthogonalisation"},
        "fp64_preconditioned": {"solve_ms": round(t64p, 3), "iters": info64p[0]["iters"],
                                "n_matvec": info64p[0]["n_matvec"],
                                "converged": info64p[0]["converged"],
                                "precision_only_speedup": round(t64p / ms, 3),
                                "note": "same preconditioner and rtol, FP64-accuracy operator throughout: "
                                        "the equal-accuracy comparison of the precision modes"},
        "fp64_plain": {"solve_ms": round(t64, 3), "iters": info64[0]["iters"],
                       "n_matvec": info64[0]["n_matvec"], "rel_residual": info64[0]["rel_residual"],
                       "converged": info64[0]["converged"], "speedup": round(t64 / ms, 3),
                       "note": "no preconditioner: the paper's plain FP64 GMRES on the GPU"},
        "mixed_unpreconditioned": {"solve_ms": round(tnp, 3), "iters": infonp[0]["iters"],
                                   "n_matvec": infonp[0]["n_matvec"],
                                   "converged": infonp[0]["converged"]},
        "precond": {"overlap_mesh_cells": PC_OVERLAP, "factor_entries": pc_elems,
                    "subdomain_total": pc_subtot, "max_subdomain": pc_nmax,
                    "apply_ms": round(pc_avg, 5) if pc_n else None,
                    "apply_gbs": round(pc_achieved, 1) if pc_n else None,
                    "apply_frac": round(pc_achieved / hbm, 4) if pc_n else None,
                    "alg_bytes_per_apply": alg_pc},
        "matvec": {"fp32_ms": round(mv32, 4), "fp32_gbs": round(bytes32 / mv32 / 1e6, 1),
                   "fp64_ms": round(mv64, 4), "fp64_gbs": round(bytes64 / mv64 / 1e6, 1),
                   "alg_bytes_fp32": bytes32, "alg_bytes_fp64": bytes64},
        "roofline": {"kernel": bin_kernel,
                     "bound": "hbm",
                     "achieved": round(achieved, 1), "peak": hbm, "unit": "GB/s",
                     "frac": round(achieved / hbm, 4), "peak_kind": peak_kind,
                     "traffic": round(traffic) if traffic else None,
                     "traffic_kind": ("scaled: ncu DRAM bytes per stored bin of the 12x12 capture x the "
                                      "stored bins here (each stored slab is streamed exactly once)"
                                      if traffic else "not captured for this kernel"),
                     "alg_bytes_per_launch": alg_bin,
                     "avg_launch_ms": round(bin_avg, 5), "launches_timed": bin_n_timed},
        "phases_ms_per_solve": {"binmul32": round(bin_ms, 3),
                                "macromodel32": round(mm_ms, 3),
                                "fft32": round(fft_ms, 3),
                                "binmul64+macromodel64": round(bin64_ms, 3),
                                "fft64+split64": round(fft64_ms + mm64_ms, 3),
                                "arnoldi": round(arn_ms, 3),
                                "scatter": round(sct_ms, 3),
                                "precond": round(pc_ms, 3),
                                "note": "one extra profiled solve outside the timed region (events add host work)"},
        "cpu_baseline": cpu,
        "e2e": {"value": round(e2e_ms, 3), "unit": "ms", "h2d_bytes_per_step": int(V.numel() * 16),
                "d2h_bytes_per_step": int(V.numel() * 16)},
        "gpu_launches": int(launches),
        "clocks": clk,
        "mirror_orbits": orbits,
        "precond_int8": pc8,
        "multi_rhs": multi,
        "accuracy": accuracy,
        "batched": batched,
        "largest": largest,
        "cpu_fft": cpu_fft,
        "serve": serve,
        "setup": setup,
        "device_bytes": dev_bytes,
    }
    print(json.dumps(out), flush=True)
    if _ABANDONED:
        # a server still holds a request that did not end: leave without
        # the teardown that would wait for it
        sys.stderr.flush()
        os._exit(0)
    if dist:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
