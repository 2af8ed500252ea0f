#!/usr/bin/env python3
"""Benchmark of the sparse hot path on one node; prints ONE JSON line.

Step = one SpMV y = A x in every format (CSR, ELL, COO, hybrid) and value
type (FP64, FP32 values+vectors) on the four synthetic matrices of the SpMV
sweep: 3D 27-point stencil 128^3 (n = 2,097,152, nnz = 55,742,968), the
power-law matrix n = 10^6 (Zipf(2) row lengths clipped to [1, 10^4]), its
mean-16 variant (row lengths clip(ceil(2.65 Z), 1, 10^4), nnz 16,016,318)
and the banded matrix n = 10^6 (half-bandwidth 64, fill 0.3).  ELL on the
power-law matrices is rejected by the padding limit and is not part of the
step.
SELL-P (slices of 64 rows) is timed the same way after the step and reported
under `extra_formats`, outside `value` (the sweep's formats are CSR, ELL, COO
and hybrid); on the power-law matrix it is rejected by the padding limit too.
CSR and COO plan parameters are chosen by the library's plan autotuner
(gko_matrix_tune, kernel kept) at setup, untimed; the plans are listed in
config.tuned_plans.
value = algorithmic bytes of all SpMVs / their summed device time (GB/s);
L2 is flushed (256 MB write) before every SpMV.  Matrices stay resident in
HBM; `e2e` repeats the step through the same C ABI calls with x copied in
from pinned host memory and y copied back inside the timed region.

--impl reference times the CPU oracle (plain C, FP64, OpenMP over rows) on
a bounded sample of the same workload on the host cores.
Multi-GPU (torchrun): every rank runs an independent replica (the SpMV
sweep has no exchange step); value is the sum over ranks of bytes divided by
the slowest rank's time.
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

METRIC = "SpMV GB/s (% HBM peak) per format; solves/s + p99 latency at 1e-8 residual, mixed vs FP64"
# power-law "mean ~16" variant: row lengths clip(ceil(lambda * Zipf(2)), 1, 1e4); lambda = 2.65 gives mean
# 16.02 (nnz 16,016,318) at seed 0
POWERLAW16_LAMBDA = 2.65
WORKLOAD = ("SpMV format sweep: CSR/ELL/COO/hybrid x FP64/FP32 (int32 indices) on 27-pt stencil 128^3, "
            "power-law n=1e6 (Zipf s=2, clip [1,1e4], seed 0), power-law-16 n=1e6 (lambda 2.65, mean 16.0), "
            "banded n=1e6 (hb 64, fill 0.3, seed 0)")
FALLBACK_HBM_GBS = 6800.0
SWEEP_FORMATS = ("csr", "ell", "coo", "hybrid")
EXTRA_FORMATS = ("sellp",)  # timed the same way, reported beside the sweep, not part of `value`


def env_rank():
    return (int(os.environ.get("RANK", 0)), int(os.environ.get("WORLD_SIZE", 1)),
            int(os.environ.get("LOCAL_RANK", 0)))


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return float(d.get("hbm_gbs", FALLBACK_HBM_GBS)), "measured"
    return FALLBACK_HBM_GBS, "fallback"


def workload_matrices(small=False):
    from paper_2006_14290_gb300 import inputs as I

    st = ("stencil27_96", I.stencil3d_27pt(96)) if small else ("stencil27_128", I.stencil3d_27pt(128))
    return [st, ("powerlaw_1m", I.powerlaw(1_000_000, seed=0)),
            ("powerlaw16_1m", I.powerlaw(1_000_000, seed=0, lam=POWERLAW16_LAMBDA)),
            ("banded_1m", I.banded(1_000_000, 64, 0.3, seed=0))]


def spmv_bytes(fmt, n_rows, n_cols, nnz, ell_nnz, tail_nnz, sv, sx, sy):
    """Algorithmic bytes of one y = A x (beta = 0): values + indices once,
    x once, y written once; padding, x re-reads and misses excluded."""
    if fmt == "csr":
        return nnz * (sv + 4) + 4 * (n_rows + 1) + sx * n_cols + sy * n_rows
    if fmt in ("ell", "sellp"):
        return nnz * (sv + 4) + sx * n_cols + sy * n_rows
    if fmt == "coo":
        return nnz * (sv + 8) + sx * n_cols + sy * n_rows
    return ell_nnz * (sv + 4) + tail_nnz * (sv + 8) + sx * n_cols + sy * n_rows


class ClockSampler:
    """nvidia-smi clocks and throttle reasons, sampled during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                                          "-i", str(self.gpu), "-lms", "100"], stdout=subprocess.PIPE,
                                         stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except Exception:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"], "samples": 0}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.thread.join(timeout=2)
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


def gpu_index(local_rank):
    vis = os.environ.get("CUDA_VISIBLE_DEVICES", "")
    ids = [v for v in vis.split(",") if v.strip()]
    if local_rank < len(ids) and ids[local_rank].strip().isdigit():
        return int(ids[local_rank])
    return local_rank


# Sources that define the SpMV kernels, their launch plans and the matrix
# layouts: the DRAM traffic recorded in profiles/traffic.json holds while
# these are unchanged (solver-only changes do not void it).
SPMV_SOURCES = ("common.cuh", "tma.cuh", "reduce.cuh", "spmv.cuh", "spmv_kernels.cuh", "spmv.cu",
                "spmv_f64.cu", "spmv_f32.cu", "spmv_bf16.cu", "matrix.cu")


def source_hash():
    h = hashlib.sha256()
    d = os.path.join(ROOT, "paper_2006_14290_gb300", "csrc")
    for f in SPMV_SOURCES:
        with open(os.path.join(d, f), "rb") as fh:
            h.update(f.encode() + fh.read())
    return h.hexdigest()[:16]


def traffic_record():
    """DRAM bytes per launch from a committed ncu summary, if it was taken on
    the current kernel sources (else None)."""
    p = os.path.join(ROOT, "profiles", "traffic.json")
    if not os.path.exists(p):
        return None
    with open(p) as f:
        d = json.load(f)
    if d.get("source_hash") != source_hash():
        return None
    return d


LINE_MAX = 3000  # characters: what a reader of the last lines of the output still gets whole


def summary_line(result):
    """The JSON line on standard output: the headline and a short form of each
    leg.  The full record (22,000 characters) goes to standard error."""
    keys = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
            "vs_baseline", "dtype", "data", "roofline", "e2e", "clocks", "gpu_launches", "cpu_baseline")
    line = {k: result[k] for k in keys if k in result}
    line["config"] = {k: v for k, v in result["config"].items() if k not in ("tuned_plans", "skipped")}
    if "cpu_baseline" in line:
        line["cpu_baseline"] = {k: v for k, v in line["cpu_baseline"].items() if k != "cores_all"}
    solvers = result.get("solvers", {})
    short = {k: v["time_ms"] for k, v in solvers.items() if isinstance(v, dict) and "time_ms" in v}
    short.update({f"batch4096_{k}": v["time_ms"] for k, v in solvers.get("batched_cg", {}).items()
                  if isinstance(v, dict) and "time_ms" in v})
    if short:
        line["solvers_ms"] = short
    serving = {k: [v["converged"], v["p99_ms"], v["solves_per_s"]] for k, v in result.get("serving", {}).items()
               if isinstance(v, dict) and "p99_ms" in v}
    if serving:
        line["serving_converged_p99ms_per_s"] = serving
    line["full_record"] = "standard error"
    for drop in ("serving_converged_p99ms_per_s", "solvers_ms"):
        if len(json.dumps(line)) <= LINE_MAX:
            break
        line.pop(drop, None)
    return json.dumps(line)


# ----------------------------------------------------------------- solvers --

def oracle_solver_sample(solver, A, b, iters, pc=False, bs=0):
    """The oracle's FP64 solve (as it stands: OpenMP over rows in its SpMV,
    vector operations sequential) run for a bounded number of iterations
    (tolerance 0 never stops early): ms per iteration on the host cores.
    bs > 0: block-Jacobi with blocks of bs rows (its setup inside the time)."""
    import oracle as O

    t0 = time.perf_counter()
    if bs:
        _, r = O.solve_block_jacobi(solver, A, b, bs, tol=0.0, maxit=iters)
    elif pc:
        _, r = O.solve_jacobi(solver, A, b, tol=0.0, maxit=iters)
    else:
        _, r = O.solve(solver, A, b, tol=0.0, maxit=iters)
    dt = time.perf_counter() - t0
    return dt * 1e3 / max(r.iterations, 1), int(r.iterations)


def cfg1_suite(G, dev, stream, flush, cores):
    """The 2D 5-point Laplacian 64^2 (n = 4,096, nnz = 20,224) with x and b
    uniform in [-1, 1] from default_rng(0) (x first): CSR FP64 SpMV (median of
    20, L2 flushed before each) and CG to 1e-10 (median of 10 solves), with the
    oracle's SpMV and CG timed beside them on 1 core and on all cores."""
    import torch
    import oracle as O
    from paper_2006_14290_gb300 import inputs as I

    A, x, b = I.laplace2d_problem(64)
    M = G.from_csr(A)
    xd = torch.from_numpy(x).to(dev)
    yd = torch.zeros(A.n_rows, dtype=torch.float64, device=dev)
    bd = torch.from_numpy(b).to(dev)
    for _ in range(3):
        G.gko_spmv(1.0, M, xd, 0.0, yd, stream=stream)
    ts = []
    for k in range(20):
        flush.fill_(float(k))
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        G.gko_spmv(1.0, M, xd, 0.0, yd, stream=stream)
        e1.record(stream)
        torch.cuda.synchronize()
        ts.append(e0.elapsed_time(e1))
    spmv_ms = float(np.median(ts))
    nb = spmv_bytes("csr", A.n_rows, A.n_cols, A.nnz, 0, 0, 8, 8, 8)
    for _ in range(3):
        xs = torch.zeros_like(bd)
        G.gko_solve_cg(M, bd, xs, 1e-10, 5000, stream=stream)
    cg_ms, res = [], None
    for _ in range(10):
        xs = torch.zeros_like(bd)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        res = G.gko_solve_cg(M, bd, xs, 1e-10, 5000, stream=stream)
        e1.record(stream)
        torch.cuda.synchronize()
        cg_ms.append(e0.elapsed_time(e1))
    out = {"n": int(A.n_rows), "nnz": int(A.nnz),
           "spmv_us": round(spmv_ms * 1e3, 2), "spmv_GB_s": round(nb / (spmv_ms * 1e-3) / 1e9, 1),
           "cg_status": int(res.status), "cg_iterations": int(res.iterations),
           "cg_rel_residual": float(res.rel_residual), "cg_ms": round(float(np.median(cg_ms)), 3),
           "cg_solves_per_s": round(1e3 / float(np.median(cg_ms)), 1)}
    orc = {}
    for tag, t in (("cores_1", 1), ("cores_all", cores)):
        used = O.set_threads(t)
        reps, t0 = 0, time.perf_counter()
        while reps < 2000 and time.perf_counter() - t0 < 1.0:
            O.spmv_csr(A, x)
            reps += 1
        sp = (time.perf_counter() - t0) / reps
        creps, t0 = 0, time.perf_counter()
        while creps < 50 and time.perf_counter() - t0 < 2.0:
            _, ro = O.cg(A, b, tol=1e-10, maxit=5000)
            creps += 1
        cg = (time.perf_counter() - t0) / creps
        orc[tag] = {"threads": used, "spmv_us": round(sp * 1e6, 2), "spmv_GB_s": round(nb / sp / 1e9, 2),
                    "cg_ms": round(cg * 1e3, 3), "cg_iterations": int(ro.iterations),
                    "cg_solves_per_s": round(1.0 / cg, 2)}
    O.set_threads(cores)
    out["oracle"] = orc
    return out


def fma_peak(G, dev, fp64=True):
    """FMA rate of the GPU measured with the library's probe (gko_bench_fma:
    8 register-resident FMA chains per thread, 8 resident 256-thread blocks
    per SM): FMAs per second from the difference of two loop counts."""
    import torch

    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    n = sms * 8 * 256
    t = torch.ones(n, dtype=torch.float64 if fp64 else torch.float32, device=dev)
    lo, hi = (1024, 3072) if fp64 else (16384, 49152)
    G.gko_bench_fma(t, lo)
    best = {}
    for loops in (lo, hi):
        ts = []
        for _ in range(3):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            G.gko_bench_fma(t, loops)
            e1.record()
            torch.cuda.synchronize()
            ts.append(e0.elapsed_time(e1))
        best[loops] = min(ts)
    return 8.0 * n * (hi - lo) / ((best[hi] - best[lo]) * 1e-3)


def gather_peak(G, dev, fp64=True, log2_len=20):
    """Random-gather rate of the GPU measured with the library's probe
    (gko_bench_gather: 8 independent LCG index streams per thread, 8 resident
    256-thread blocks per SM, one element per gather from an L2-resident
    vector of 2^20 elements, the power-law matrices' x): gathers per second
    from the difference of two loop counts."""
    import torch

    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    n = sms * 8 * 256
    dt = torch.float64 if fp64 else torch.float32
    x = torch.rand(1 << log2_len, dtype=dt, device=dev)
    out = torch.empty(n, dtype=dt, device=dev)
    lo, hi = 32, 96
    G.gko_bench_gather(x, out, lo)
    best = {}
    for loops in (lo, hi):
        ts = []
        for _ in range(3):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            G.gko_bench_gather(x, out, loops)
            e1.record()
            torch.cuda.synchronize()
            ts.append(e0.elapsed_time(e1))
        best[loops] = min(ts)
    return 8.0 * n * (hi - lo) / ((best[hi] - best[lo]) * 1e-3)


def solver_suite(G, dev, stream, flush=None, oracle_cores=0):
    """Krylov solves to 1e-8 relative residual, FP64 vs mixed precision:
    CG on the 7-point Poisson problem 256^3 (b = A*1) and BiCGSTAB / GMRES(30)
    on 7-point upwind convection-diffusion 128^3 (cell Peclet 10, b = A*1);
    plus 1,000 CG iterations of fixed work (the paper's CG experiment), the
    2D 5-point 64^2 CG configuration, and the batched CG.  With oracle_cores
    > 0 every solve has the oracle's FP64 solve of the same problem timed
    beside it on a bounded sample of iterations (oracle_ms = its ms per
    iteration x the GPU's FP64 iteration count)."""
    import torch
    import oracle as O
    from paper_2006_14290_gb300 import inputs as I

    out = {}
    fp64_fma = fma_peak(G, dev)
    hbm_peak, _ = measured_peaks()
    out["fp64_fma_peak"] = {"fma_per_s": round(fp64_fma, -8), "tflops": round(2 * fp64_fma / 1e12, 3),
                            "how": "gko_bench_fma, 8 FMA chains per thread, 8 blocks of 256 per SM, "
                                   "difference of 3072 and 1024 loops"}
    if oracle_cores:
        O.lib()
        O.set_threads(oracle_cores)
    if flush is not None:
        out["cfg1_laplace64"] = cfg1_suite(G, dev, stream, flush, oracle_cores or (os.cpu_count() or 1))

    def run(tag, solver, M, bd, n, nnz, prec, maxit=20000, tol=1e-8, restart=30, pc=0, refine=0, bs=0):
        fn = {"cg": G.gko_solve_cg, "bicgstab": G.gko_solve_bicgstab, "gmres": G.gko_solve_gmres}[solver]
        if solver == "bicgstab":
            maxit = 2000
        # the library's refinement defaults (GMRES: one restart cycle per step)
        opts = G.opts(precision=prec, restart=restart, preconditioner=pc, refinement=refine, block_size=bs)
        if tag == "bicgstab_convdiff128_mixed_f32":  # known not to converge: keep it short
            opts = G.opts(precision=prec, inner_maxit=500, max_outer=3)
            maxit = 500
        xd = torch.zeros(n, dtype=torch.float64, device=dev)
        fn(M, bd, xd, tol, maxit, opts, stream=stream)  # warm-up (also builds the low-precision copy)
        xd.zero_()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        t0 = time.perf_counter()
        res = fn(M, bd, xd, tol, maxit, opts, stream=stream)
        wall = time.perf_counter() - t0
        e1.record(stream)
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1)
        sv = 8 if prec == G.PRECISION_F64 else (4 if prec == G.PRECISION_MIXED_F32 else 2)
        vb = 8 if prec == G.PRECISION_F64 else 4
        # Jacobi: d and z = d r; block-Jacobi: r, z and bs FP64 block entries per row
        bjac = pc == G.PRECOND_BLOCK_JACOBI
        per_vec_passes = {"cg": 10, "bicgstab": 16, "gmres": 2 * 30 + 6}[solver]
        per_vec_passes += (2 + bs) if bjac else 2 if pc else 0
        spmvs = {"cg": 1, "bicgstab": 2, "gmres": 1}[solver]
        it_bytes = spmvs * (nnz * (sv + 4) + 4 * (n + 1) + 2 * vb * n) + per_vec_passes * vb * n
        its = max(res.iterations, 1)
        out[tag] = {"status": int(res.status), "iterations": int(res.iterations),
                    "outer_iterations": int(res.outer_iterations), "rel_residual": float(res.rel_residual),
                    "time_ms": round(ms, 3), "wall_ms": round(wall * 1e3, 3), "solves_per_s": round(1e3 / ms, 3),
                    "GB_s_per_iteration": round(it_bytes * its / (ms * 1e-3) / 1e9, 1),
                    "frac_hbm": round(it_bytes * its / (ms * 1e-3) / 1e9 / hbm_peak, 4)}
        if prec == G.PRECISION_F64:
            # FP64 FMAs per iteration: SpMV nnz; CG x, r, p updates and the
            # p.q and r.r dots; BiCGSTAB p (2), s, x (2), r updates and five
            # dots; GMRES(30) both Gram-Schmidt passes (a dot and an axpy
            # per basis vector each, mean j + 1 = 15.5) and the norm;
            # Jacobi: z = d r and r.z; block-Jacobi: bs per row for z and r.z
            fma_it = {"cg": nnz + 5 * n, "bicgstab": 2 * nnz + 12 * n, "gmres": nnz + 63 * n}[solver]
            fma_it += (bs + 1) * n if bjac else 2 * n if pc else 0
            t_fp64, t_hbm = fma_it / fp64_fma, it_bytes / (hbm_peak * 1e9)
            out[tag].update({"fp64_fmas_per_iteration": int(fma_it),
                             "frac_fp64": round(fma_it * its / (ms * 1e-3) / fp64_fma, 4),
                             "bound": "fp64" if t_fp64 > t_hbm else "hbm",
                             "frac_of_bound": round(max(t_fp64, t_hbm) * its / (ms * 1e-3), 4)})
        return ms

    def oracle_beside(tags, solver, A, b, sample_iters, pc=False, fp64_tag=None, bs=0):
        """Oracle FP64 solve of the same problem on a bounded sample; each tag
        gets oracle_ms = ms per iteration x the FP64 GPU run's iterations."""
        if not oracle_cores:
            return
        sid = {"cg": O.CG, "bicgstab": O.BICGSTAB, "gmres": O.GMRES}[solver]
        per_it, done = oracle_solver_sample(sid, A, b, sample_iters, pc=pc, bs=bs)
        its = out[fp64_tag or tags[0]]["iterations"]
        pcname = f" + block-Jacobi({bs})" if bs else " + Jacobi" if pc else ""
        for t in tags:
            out[t]["oracle_ms"] = round(per_it * its, 1)
            out[t]["oracle_sample"] = (f"oracle FP64 {solver}{pcname}: {done} iterations timed "
                                       f"({per_it:.2f} ms each, {oracle_cores} threads in its SpMV), "
                                       f"x {its} iterations of the GPU FP64 run")

    def speedup(base, other):
        """Time ratio of two runs, only when both converged (a ratio against
        a breakdown or a stalled run says nothing).  The FP64 side is the
        faster of the CSR handle and, where it was run, the ELL handle
        (base + "_ell") of the same matrix."""
        if out[other]["status"] != G.OK:
            return None
        t = [out[k]["time_ms"] for k in (base, base + "_ell") if k in out and out[k]["status"] == G.OK]
        if not t:
            return None
        return round(min(t) / out[other]["time_ms"], 3)

    A = I.stencil3d_7pt(256)
    M = G.from_csr(A)
    n, nnz = A.n_rows, A.nnz
    ones = torch.ones(n, dtype=torch.float64, device=dev)
    bd = torch.zeros_like(ones)
    G.gko_spmv(1.0, M, ones, 0.0, bd, stream=stream)
    run("cg_poisson256_f64", "cg", M, bd, n, nnz, G.PRECISION_F64)
    E = G.gko_matrix_convert_to_ell(M)
    run("cg_poisson256_f64_ell", "cg", E, bd, n, nnz, G.PRECISION_F64)
    del E
    run("cg_poisson256_mixed_f32", "cg", M, bd, n, nnz, G.PRECISION_MIXED_F32)
    run("cg_poisson256_mixed_bf16", "cg", M, bd, n, nnz, G.PRECISION_MIXED_BF16)
    run("cg_poisson256_mixed_f32_restart", "cg", M, bd, n, nnz, G.PRECISION_MIXED_F32, refine=G.REFINE_RESTART)
    out["cg_poisson256_mixed_f32_speedup"] = speedup("cg_poisson256_f64", "cg_poisson256_mixed_f32")
    out["cg_poisson256_mixed_f32_restart_speedup"] = speedup("cg_poisson256_f64", "cg_poisson256_mixed_f32_restart")
    # fixed work: 1,000 iterations (tolerance 0 never stops early)
    xd = torch.zeros(n, dtype=torch.float64, device=dev)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    res = G.gko_solve_cg(M, bd, xd, 0.0, 1000, G.opts(check_every=1000), stream=stream)
    dt = time.perf_counter() - t0
    out["cg_poisson256_1000_iterations"] = {"iterations": int(res.iterations), "time_ms": round(dt * 1e3, 3),
                                            "iterations_per_s": round(res.iterations / dt, 1)}
    if oracle_cores:
        b_host = bd.cpu().numpy()
        oracle_beside(["cg_poisson256_f64", "cg_poisson256_mixed_f32", "cg_poisson256_mixed_bf16",
                       "cg_poisson256_mixed_f32_restart"], "cg", A, b_host, 8)
        per_it = out["cg_poisson256_f64"]["oracle_ms"] / max(out["cg_poisson256_f64"]["iterations"], 1)
        out["cg_poisson256_1000_iterations"]["oracle_ms"] = round(per_it * 1000, 1)
        del b_host
    del A, M, ones, bd, xd
    for P, sfx in ((10.0, ""), (1.0, "_P1")):
        A = I.convdiff3d_7pt(128, P)
        M = G.from_csr(A)
        n, nnz = A.n_rows, A.nnz
        ones = torch.ones(n, dtype=torch.float64, device=dev)
        bd = torch.zeros_like(ones)
        G.gko_spmv(1.0, M, ones, 0.0, bd, stream=stream)
        b_host = bd.cpu().numpy()
        # unpreconditioned BiCGSTAB does not converge at cell Peclet 10 on 128^3
        # (the oracle diverges too); Peclet 1 is the converging companion case
        solvers = ("bicgstab", "gmres") if P == 10.0 else ("bicgstab",)
        for solver in solvers:
            tag = ("bicgstab" if solver == "bicgstab" else "gmres30") + "_convdiff128" + sfx
            run(f"{tag}_f64", solver, M, bd, n, nnz, G.PRECISION_F64)
            if not (solver == "bicgstab" and P == 10.0):  # the FP64 baseline in ELL too (faster of the two)
                E = G.gko_matrix_convert_to_ell(M)
                run(f"{tag}_f64_ell", solver, E, bd, n, nnz, G.PRECISION_F64)
                del E
            run(f"{tag}_mixed_f32", solver, M, bd, n, nnz, G.PRECISION_MIXED_F32)
            out[f"{tag}_mixed_f32_speedup"] = speedup(f"{tag}_f64", f"{tag}_mixed_f32")
            if solver == "bicgstab" and P == 1.0:  # the classic restarted refinement beside the default
                run(f"{tag}_mixed_f32_restart", solver, M, bd, n, nnz, G.PRECISION_MIXED_F32,
                    refine=G.REFINE_RESTART)
                out[f"{tag}_mixed_f32_restart_speedup"] = speedup(f"{tag}_f64", f"{tag}_mixed_f32_restart")
            oracle_beside([t for t in (f"{tag}_f64", f"{tag}_mixed_f32", f"{tag}_mixed_f32_restart") if t in out],
                          solver, A, b_host, 30 if solver == "gmres" else 12)
        del A, M, ones, bd, b_host
    # Jacobi preconditioning on the variable-coefficient Poisson problem 128^3
    # (coefficients exp(N(0,1)) per cell, default_rng(0); b = A*1)
    A = I.varcoef3d_7pt(128, np.random.default_rng(0))
    M = G.from_csr(A)
    n, nnz = A.n_rows, A.nnz
    ones = torch.ones(n, dtype=torch.float64, device=dev)
    bd = torch.zeros_like(ones)
    G.gko_spmv(1.0, M, ones, 0.0, bd, stream=stream)
    run("cg_varcoef128_f64", "cg", M, bd, n, nnz, G.PRECISION_F64)
    run("cg_varcoef128_jacobi_f64", "cg", M, bd, n, nnz, G.PRECISION_F64, pc=G.PRECOND_JACOBI)
    run("cg_varcoef128_jacobi_mixed_f32", "cg", M, bd, n, nnz, G.PRECISION_MIXED_F32, pc=G.PRECOND_JACOBI)
    # block-Jacobi: blocks of 8 consecutive rows (x-line segments of the grid)
    run("cg_varcoef128_bjacobi8_f64", "cg", M, bd, n, nnz, G.PRECISION_F64, pc=G.PRECOND_BLOCK_JACOBI, bs=8)
    run("cg_varcoef128_bjacobi8_mixed_f32", "cg", M, bd, n, nnz, G.PRECISION_MIXED_F32, pc=G.PRECOND_BLOCK_JACOBI,
        bs=8)
    out["cg_varcoef128_jacobi_speedup"] = speedup("cg_varcoef128_f64", "cg_varcoef128_jacobi_f64")
    out["cg_varcoef128_jacobi_mixed_f32_speedup"] = speedup("cg_varcoef128_f64", "cg_varcoef128_jacobi_mixed_f32")
    out["cg_varcoef128_bjacobi8_speedup"] = speedup("cg_varcoef128_f64", "cg_varcoef128_bjacobi8_f64")
    out["cg_varcoef128_bjacobi8_mixed_f32_speedup"] = speedup("cg_varcoef128_f64", "cg_varcoef128_bjacobi8_mixed_f32")
    if oracle_cores:
        b_host = bd.cpu().numpy()
        oracle_beside(["cg_varcoef128_f64"], "cg", A, b_host, 12)
        oracle_beside(["cg_varcoef128_jacobi_f64", "cg_varcoef128_jacobi_mixed_f32"], "cg", A, b_host, 12, pc=True)
        oracle_beside(["cg_varcoef128_bjacobi8_f64", "cg_varcoef128_bjacobi8_mixed_f32"], "cg", A, b_host, 12,
                      bs=8)
        del b_host
    del A, M, ones, bd
    out["batched_cg"] = batched_suite(G, dev, stream, oracle_cores, fp64_fma)
    return out


# nominal FP64 rate of the part (2 FMA per SM per clock, 152 SMs, 2.07 GHz)


def batched_suite(G, dev, stream, oracle_cores=0, fp64_fma=None):
    """4096 variable-coefficient 2D 5-point systems (sides log-uniform in
    [8, 64]) solved by batched CG to 1e-10 in one persistent graph-captured
    launch; FP64 and FP32 storage; schedule from the autotuner.  Work per
    batch: global bytes = sum over systems of iterations x (values, columns
    and row pointers of the system's matrix + x read and written; r, p, q live
    in shared memory), FP64 FMAs = sum of iterations x (nnz + 5 n).  The
    oracle's batched CG (OpenMP over systems) is timed beside it."""
    import torch
    from paper_2006_14290_gb300 import inputs as I

    sides = I.batch_sides(4096)
    systems, bs = [], []
    for i, sd in enumerate(sides):
        A, b = I.batch_system(i, int(sd))
        systems.append(A)
        bs.append(b)
    b = torch.from_numpy(np.concatenate(bs)).to(dev)
    rows = np.array([S.n_rows for S in systems], np.int64)
    nnzs = np.array([S.nnz for S in systems], np.int64)
    res = {"systems": 4096, "rows": int(rows.sum()), "nnz": int(nnzs.sum())}
    peak_hbm, _ = measured_peaks()
    for storage, tag, mixed in ((G.F64, "f64", False), (G.F32, "f32_storage", False), (G.F64, "mixed_f32", True)):
        B = G.Batch(systems, storage=storage)
        if mixed:
            B.set_precision(G.PRECISION_MIXED_F32)
        x0 = torch.zeros(B.total_rows, dtype=torch.float64, device=dev)
        tuned = B.tune(b, x0, 1e-10, 20000, stream=stream)
        x = torch.zeros_like(x0)
        B.cg(b, x, 1e-10, 20000, stream=stream)  # capture the graph
        times = []
        for _ in range(3):
            x.zero_()
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            code, it, rr, st = B.cg(b, x, 1e-10, 20000, stream=stream)
            e1.record(stream)
            torch.cuda.synchronize()
            times.append(e0.elapsed_time(e1))
        ms = float(np.median(times))
        sv = 8 if storage == G.F64 and not mixed else 4
        itd = it.astype(np.float64)
        up = B.last_updates().astype(np.float64)
        # mixed: FP32 values in the recurrences (x stays in global memory only
        # at updates), two FP64 FMAs per row and iteration (the dots), and per
        # update an FP64 product with the stored values plus its residual norm
        nbytes = float(np.sum(itd * (nnzs * (sv + 4) + 4 * (rows + 1) + (0 if mixed else 16) * rows)))
        if mixed:
            nbytes += float(np.sum(up * (nnzs * 12 + 4 * (rows + 1) + 32 * rows)))
            fmas = float(np.sum(itd * 2 * rows + up * (nnzs + 2 * rows)))
        else:
            fmas = float(np.sum(itd * (nnzs + 5 * rows)))
        fp64_fma = fp64_fma or fma_peak(G, dev)
        fp64_frac = fmas / (ms * 1e-3) / fp64_fma
        res[tag] = {"status": int(code), "time_ms": round(ms, 3), "systems_per_s": round(4096 / (ms * 1e-3), 1),
                    "schedule": tuned,
                    "tuned_over": "no schedule: every system is solved resident on an SM" if mixed
                    else "warp rows {0,64,144,256} x threads {256,512,1024} x CSR/ELL",
                    "iterations_total": int(it.sum()), "iterations_max": int(it.max()),
                    "max_rel_residual": float(rr.max()), "bytes": nbytes, "fp64_fmas": fmas,
                    "GB_s": round(nbytes / (ms * 1e-3) / 1e9, 1),
                    "frac_hbm": round(nbytes / (ms * 1e-3) / 1e9 / peak_hbm, 4),
                    "frac_fp64": round(fp64_frac, 4),
                    "fp64_peak": f"{2 * fp64_fma / 1e12:.3f} TFLOP/s measured (gko_bench_fma)"}
        if mixed:
            res[tag]["updates_total"] = int(up.sum())
            res[tag]["note"] = ("reliable-update CG per system: FP32 recurrences, FP64 dots and x, "
                                "replaced residuals with the FP64 values")
        del B
    if oracle_cores:
        import oracle as O

        O.set_threads(oracle_cores)
        t0 = time.perf_counter()
        _, oit, orr, ost = O.batch_cg(systems, bs, tol=1e-10, maxit=20000)
        dt = time.perf_counter() - t0
        res["oracle"] = {"ms": round(dt * 1e3, 1), "systems_per_s": round(4096 / dt, 1), "threads": oracle_cores,
                         "converged": int(np.sum(ost == 0)), "iterations_total": int(oit.sum()),
                         "sample": "the full batch: the oracle's FP64 CG per system, OpenMP over systems"}
        res["f64"]["oracle_ms"] = res["oracle"]["ms"]
        res["f32_storage"]["oracle_ms"] = res["oracle"]["ms"]
        t0 = time.perf_counter()
        _, oit, oup, orr, ost = O.batch_cg_reliable(systems, bs, tol=1e-10, maxit=20000)
        dt = time.perf_counter() - t0
        res["oracle_mixed"] = {"ms": round(dt * 1e3, 1), "systems_per_s": round(4096 / dt, 1),
                               "threads": oracle_cores, "converged": int(np.sum(ost == 0)),
                               "iterations_total": int(oit.sum()), "updates_total": int(oup.sum()),
                               "sample": "the full batch: the oracle's reliable-update CG per system, "
                                         "OpenMP over systems"}
        res["mixed_f32"]["oracle_ms"] = res["oracle_mixed"]["ms"]
    res["mixed_f32_speedup"] = (round(res["f64"]["time_ms"] / res["mixed_f32"]["time_ms"], 3)
                                if res["f64"]["status"] == G.OK and res["mixed_f32"]["status"] == G.OK else None)
    return res


# ----------------------------------------------------------------- serving --

SERVING_RATES = (100.0, 250.0, 500.0, 1000.0, 2000.0)


def serving_suite(G, rates=SERVING_RATES, per_type=64, slots=8, budget_bytes=150 << 30, max_requests=500):
    """Poisson arrivals of sparse solves against resident matrices.

    Pool: `per_type` variable-coefficient 7-point Poisson matrices (CG, Jacobi
    preconditioned, as the variable coefficients call for) and `per_type`
    upwind convection-diffusion matrices with cell Peclet ~ U[1, 20]
    (BiCGSTAB), cube sides rint(n^(1/3)) for n log-uniform in [1e3, 4e6], all
    from default_rng(0), uploaded before any window.  Requests: one Poisson
    stream from default_rng(1) (70% CG / 30% BiCGSTAB, uniformly chosen pool
    matrix), each with its own right-hand side b = A v, v uniform in [0.5,
    1.5] from default_rng([2, request]); tolerance 1e-8, iteration caps CG
    5000, BiCGSTAB 500; admitted by a 150 GB budget over `slots` concurrent
    solves.  Every rate replays the same requests with arrival times scaled
    to it (window: the first min(max_requests, rate) arrivals, at most 1 s),
    FP64 and mixed FP32.  Every request that does not return GKO_OK is listed
    with its status, solver, matrix, size, iterations and residual.
    """
    import torch
    from paper_2006_14290_gb300 import inputs as I

    rng = np.random.default_rng(0)
    pool = []
    for kind in ("cg", "bicgstab"):
        for _ in range(per_type):
            n = float(np.exp(rng.uniform(np.log(1e3), np.log(4e6))))
            side = max(4, int(np.rint(n ** (1.0 / 3.0))))
            if kind == "cg":
                A = I.varcoef3d_7pt(side, rng)
            else:
                A = I.convdiff3d_7pt(side, float(rng.uniform(1.0, 20.0)))
            pool.append([kind, G.from_csr(A), int(A.n_rows), side])
            del A
    arr = np.random.default_rng(1)
    unit_times = np.cumsum(arr.exponential(1.0, max_requests))  # arrivals at rate 1
    picks = []
    for _ in range(max_requests):
        k = 0 if arr.random() < 0.7 else 1
        picks.append(int(arr.integers(0, per_type)) + per_type * k)
    bs = []
    for r, m in enumerate(picks):
        n = pool[m][2]
        v = torch.from_numpy(np.random.default_rng([2, r]).uniform(0.5, 1.5, n)).cuda()
        bd = torch.zeros_like(v)
        G.gko_spmv(1.0, pool[m][1], v, 0.0, bd)
        bs.append(bd.cpu().numpy())
        del v, bd
    out = {"pool_matrices": len(pool), "pool_rows_total": int(sum(p[2] for p in pool)), "slots": slots,
           "budget_GB": budget_bytes / 2**30, "rates": list(rates)}
    for rate in rates:
        count = int(min(max_requests, np.searchsorted(unit_times / rate, 1.0, side="right")))
        times = unit_times[:count] / rate
        for prec_name, prec in (("f64", G.PRECISION_F64), ("mixed_f32", G.PRECISION_MIXED_F32)):
            S = G.Server(slots=slots, budget_bytes=budget_bytes)
            ids = [S.add_matrix(p[1]) for p in pool]
            opts = G.opts(precision=prec, inner_maxit=1000)
            opts_cg = G.opts(precision=prec, inner_maxit=1000, preconditioner=G.PRECOND_JACOBI)
            t0 = time.perf_counter()
            rids = []
            for r in range(count):
                now = time.perf_counter() - t0
                if times[r] > now:
                    time.sleep(times[r] - now)
                m = picks[r]
                cg = pool[m][0] == "cg"
                rids.append(S.submit(ids[m], 0 if cg else 1, bs[r], 1e-8, 5000 if cg else 500,
                                     opts_cg if cg else opts))
            results = [S.result(q) for q in rids]
            wall = time.perf_counter() - t0
            st = S.stats()
            S.close()
            failed = []
            for r, (code, res, _, lat) in enumerate(results):
                if code != G.OK:
                    m = picks[r]
                    failed.append({"request": r, "status": int(code), "solver": pool[m][0], "matrix": m,
                                   "n": pool[m][2], "iterations": int(res.iterations),
                                   "rel_residual": float(res.rel_residual)})
            cg_req = sum(1 for r in range(count) if pool[picks[r]][0] == "cg")
            out[f"rate{int(rate)}_{prec_name}"] = {
                "requests": count, "window_s": round(float(times[-1]), 3) if count else 0.0,
                "converged": count - len(failed), "cg_requests": cg_req,
                "cg_converged": cg_req - sum(1 for f in failed if f["solver"] == "cg"),
                "p50_ms": round(st["p50_ms"], 3), "p99_ms": round(st["p99_ms"], 3),
                "solves_per_s": round(st["solves_per_s"], 2), "drain_s": round(wall, 3),
                "peak_concurrent": st["peak_active"], "failed": failed}
    return out


# ------------------------------------------------ subwarp microbenchmark --

def subwarp_microbench(G, dev, stream):
    """Section 3.3 method: time of 1000 subwarp reductions = t(2000 inner
    loops) - t(1000), median of 5, for the library primitive, CUDA
    cooperative groups and the full-warp shuffle, subwarp sizes 4..32, on
    4 blocks of 256 threads per SM; ratio S=4 / S=32 against log2(4)/log2(32)."""
    import torch

    props = torch.cuda.get_device_properties(dev)
    n = 256 * 4 * props.multi_processor_count
    out = {"threads": n, "theory_ratio_4_over_32": round(2 / 5, 3)}
    for dt in (torch.float32, torch.float64):
        data = torch.zeros(n, dtype=dt, device=dev)
        for impl, iname in ((0, "library"), (1, "cooperative_groups"), (2, "legacy_shfl")):
            per = {}
            for S in (4, 8, 16, 32):
                diffs = []
                for _ in range(5):
                    t = []
                    for loops in (1000, 2000):
                        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                        a.record(stream)
                        G.gko_bench_subwarp_reduce(S, impl, data, loops, stream=stream)
                        b.record(stream)
                        torch.cuda.synchronize()
                        t.append(a.elapsed_time(b))
                    diffs.append(t[1] - t[0])
                per[S] = statistics.median(diffs) * 1e3  # us per 1000 reductions
            out[f"{'f32' if dt == torch.float32 else 'f64'}/{iname}"] = {
                "us_per_1000": {str(k): round(v, 2) for k, v in per.items()},
                "ratio_4_over_32": round(per[4] / per[32], 3) if per[32] > 0 else None}
    return out


# ------------------------------------------------------ cuSPARSE context --

def cusparse_context(mats, dev, stream, flush, steps, peak):
    """cuSPARSE CSR SpMV (torch.sparse CSR @ x, int32 indices) on the sweep
    matrices, timed like the sweep (L2 flushed, CUDA events): an outside
    reference point on the same GPU, not an oracle and not part of `value`."""
    import torch

    out = {}
    for name, A in mats:
        crow = torch.from_numpy(A.row_ptr.astype(np.int32)).to(dev)
        col = torch.from_numpy(A.col.astype(np.int32)).to(dev)
        for dt, tdt, sv in (("f64", torch.float64, 8), ("f32", torch.float32, 4)):
            try:
                val = torch.from_numpy(A.val).to(dev, tdt)
                M = torch.sparse_csr_tensor(crow, col, val, (A.n_rows, A.n_cols))
                x = torch.from_numpy(np.random.default_rng(1).uniform(-1, 1, A.n_cols)).to(dev, tdt)
                for _ in range(3):
                    y = M @ x
                ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
                      for _ in range(steps)]
                for k in range(steps):
                    flush.fill_(float(k))
                    ev[k][0].record(stream)
                    y = M @ x
                    ev[k][1].record(stream)
                torch.cuda.synchronize()
                ms = sum(a.elapsed_time(b) for a, b in ev) / steps
                nb = spmv_bytes("csr", A.n_rows, A.n_cols, A.nnz, 0, 0, sv, sv, sv)
                out[f"{name}/csr/{dt}"] = {"ms": round(ms, 4), "GB_s": round(nb / (ms * 1e-3) / 1e9, 1),
                                           "frac": round(nb / (ms * 1e-3) / 1e9 / peak, 4)}
                del M, val, x, y
            except (RuntimeError, TypeError) as e:
                out[f"{name}/csr/{dt}"] = {"unavailable": str(e).splitlines()[0][:160]}
        del crow, col
    return {"library": "cuSPARSE CSR SpMV through torch.sparse_csr_tensor @ x (torch " + torch.__version__ + ")",
            "cases": out}


# --------------------------------------------------------------- reference --

def run_reference(args):
    rank, world, _ = env_rank()
    if rank != 0:
        return
    import oracle as O

    O.lib()
    cores = O.set_threads(os.cpu_count() or 1)
    mats = workload_matrices()
    step_bytes = 0
    for name, A in mats:
        step_bytes += spmv_bytes("csr", A.n_rows, A.n_cols, A.nnz, 0, 0, 8, 8, 8)
    xs = {name: np.random.default_rng(0).uniform(-1, 1, A.n_cols) for name, A in mats}

    def one_step():
        for name, A in mats:
            O.spmv_csr(A, xs[name])

    for _ in range(args.warmup):
        one_step()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        one_step()
    dt = time.perf_counter() - t0
    gbs = step_bytes * args.steps / dt / 1e9
    sample = (f"oracle FP64 CSR SpMV on the {len(mats)} sweep matrices per step ({args.steps} steps after "
              f"{args.warmup} warm-up), OpenMP over rows on {cores} threads")
    line = {"impl": "reference", "metric": METRIC, "value": round(gbs, 3), "unit": "GB/s", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(dt * 1e3 / args.steps, 3),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": WORKLOAD, "l2": "host caches (CPU run)"},
            "cpu_baseline": {"value": round(gbs, 3), "unit": "GB/s", "cores": cores, "kind": "oracle",
                             "sample": sample},
            "e2e": {"value": round(gbs, 3), "unit": "GB/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def cpu_baseline(mats, budget_s=12.0):
    """The oracle as it stands on the host cores, on a bounded sample: FP64
    CSR SpMV over the sweep matrices, on all cores (OpenMP over rows) and on
    one core."""
    import oracle as O

    O.lib()
    xs = {name: np.random.default_rng(0).uniform(-1, 1, A.n_cols) for name, A in mats}
    out = {}
    for tag, threads, budget in (("cores_all", os.cpu_count() or 1, budget_s), ("cores_1", 1, budget_s / 2)):
        cores = O.set_threads(threads)
        nbytes, reps = 0, 0
        t0 = time.perf_counter()
        while reps < 20 and (time.perf_counter() - t0) < budget:
            for name, A in mats:
                O.spmv_csr(A, xs[name])
                nbytes += spmv_bytes("csr", A.n_rows, A.n_cols, A.nnz, 0, 0, 8, 8, 8)
            reps += 1
        dt = time.perf_counter() - t0
        out[tag] = {"value": round(nbytes / dt / 1e9, 3), "cores": cores, "passes": reps, "s": round(dt, 2)}
    O.set_threads(os.cpu_count() or 1)
    allc = out["cores_all"]
    return {"value": allc["value"], "unit": "GB/s", "cores": allc["cores"], "kind": "oracle",
            "sample": (f"FP64 CSR SpMV on the {len(mats)} sweep matrices, {allc['passes']} passes "
                       f"({allc['s']:.1f} s) with OpenMP over rows; one-core figure in cores_1"),
            "cores_all": out["cores_all"], "cores_1": out["cores_1"]}


# ------------------------------------------------------------ multi-rank --

def ranks_max(values, device):
    """Element-wise maximum over all ranks (the slowest rank's times); the
    identity on one rank.  Works with NCCL (CUDA tensors) and gloo (CPU)."""
    import torch
    import torch.distributed as dist

    t = torch.tensor([float(v) for v in values], dtype=torch.float64, device=device)
    if dist.is_available() and dist.is_initialized() and dist.get_world_size() > 1:
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return [float(v) for v in t.cpu()]


def whole_job_gbs(world, bytes_per_rank, ms):
    """Whole-job throughput: every rank processes bytes_per_rank per step
    (replicas, weak scaling); time is the slowest rank's."""
    return world * bytes_per_rank / (ms * 1e-3) / 1e9


# ---------------------------------------------------------------- our path --

def build_cases(G, mats, dev, formats=("csr", "ell", "coo", "hybrid"), tune=True):
    """Every (matrix, format, value type) SpMV case of the sweep, resident on
    the device, with its algorithmic bytes and the number of kernel launches
    one gko_spmv call makes for it."""
    import torch

    convs = {"ell": lambda m: G.gko_matrix_convert_to_ell(m), "coo": G.gko_matrix_convert_to_coo,
             "hybrid": lambda m: G.gko_matrix_convert_to_hybrid(m), "sellp": lambda m: G.gko_matrix_convert_to_sellp(m)}
    cases, skipped = [], []
    for name, A in mats:
        M64 = G.from_csr(A)
        base = {"csr": M64} if "csr" in formats else {}
        for fmt in formats:
            if fmt == "csr":
                continue
            try:
                base[fmt] = convs[fmt](M64)
            except G.GkoError as e:
                if e.status != G.FORMAT_UNSUITABLE:
                    raise
                skipped.append(f"{name}/{fmt}: padding over the limit")
        x64 = torch.from_numpy(np.random.default_rng(1).uniform(-1, 1, A.n_cols)).to(dev)
        x32 = x64.float()
        for fmt, M in base.items():
            inf = M.info()
            for dt in ("f64", "f32"):
                H = M if dt == "f64" else G.gko_matrix_convert_values(M, G.F32)
                sv = 8 if dt == "f64" else 4
                ell_nnz = inf["nnz"] - inf["coo_nnz"] if fmt == "hybrid" else 0
                nb = spmv_bytes(fmt, A.n_rows, A.n_cols, A.nnz, ell_nnz, inf["coo_nnz"], sv, sv, sv)
                x = x64 if dt == "f64" else x32
                y = torch.zeros(A.n_rows, dtype=x.dtype, device=dev)
                plan = None
                if tune and fmt in ("csr", "coo"):  # setup step: the plan autotuner, untimed; the kernel
                    # itself stays the histogram rule's, so profiled runs launch the same kernels
                    k, S, R, cap, _ = H.tune(x, y, reps=2, keep_kernel=True)
                    plan = {"kernel": k, "subwarp": S, "rows_per_subwarp": R, "stage_cap": cap}
                coo_launches = 2 if inf["coo_nnz"] > 0 and fmt in ("coo", "hybrid") else 0
                hp = H.plan() if fmt in ("csr", "coo") else None
                csr_launches = 2 if hp and hp["kernel"] in (2, 3) else 1 + (2 if hp and hp["n_long_rows"] > 0 else 0)
                if fmt == "coo" and hp["kernel"] == 1:
                    coo_launches = 1  # row-block COO: one launch, no tile fix-up
                launches = {"csr": csr_launches, "ell": 1, "sellp": 1,
                            "coo": coo_launches if coo_launches else 1, "hybrid": 1 + coo_launches}[fmt]
                cases.append({"label": f"{name}/{fmt}/{dt}", "M": H, "x": x, "y": y, "bytes": nb, "plan": plan,
                              "launches": launches, "nnz": int(A.nnz), "xh": x.cpu().pin_memory(),
                              "yh": torch.empty(A.n_rows, dtype=x.dtype).pin_memory()})
        del A
    return cases, skipped


def profile_cases(args):
    """One SpMV per case (after one untimed pass), for ncu: prints the cases
    in launch order with their launch counts, algorithmic bytes and nnz."""
    import torch
    from paper_2006_14290_gb300 import gko as G

    G.load()
    dev = torch.device("cuda", 0)
    cases, _ = build_cases(G, workload_matrices(small=args.small), dev, formats=SWEEP_FORMATS + EXTRA_FORMATS)
    for c in cases:
        G.gko_spmv(1.0, c["M"], c["x"], 0.0, c["y"])
    torch.cuda.synchronize()
    torch.cuda.nvtx.range_push("profile_cases")
    for c in cases:
        G.gko_spmv(1.0, c["M"], c["x"], 0.0, c["y"])
    torch.cuda.synchronize()
    torch.cuda.nvtx.range_pop()
    G.gko_device_status()
    print(json.dumps([[c["label"], c["launches"], int(c["bytes"]), c["nnz"]] for c in cases]))

def profile_solvers(args):
    """Short fixed-work solves for ncu launch lists, convection-diffusion
    128^3, tolerance 0: BiCGSTAB FP64 (40 iterations, cell Peclet 1),
    BiCGSTAB mixed FP32 (one refinement step of 40 inner iterations, Peclet 1)
    and GMRES(30) FP64 (one restart cycle, Peclet 10); each runs once
    untimed, then once inside the NVTX range "profile_solvers".  With
    --precond instead: CG on the variable-coefficient Poisson problem 128^3,
    40 iterations each of Jacobi mixed FP32, block-Jacobi (blocks of 8)
    mixed FP32 and block-Jacobi FP64."""
    import torch
    from paper_2006_14290_gb300 import gko as G
    from paper_2006_14290_gb300 import inputs as I

    G.load()
    out = {}
    if args.precond:
        A = I.varcoef3d_7pt(128, np.random.default_rng(0))
        M = G.from_csr(A)
        ones = torch.ones(A.n_rows, dtype=torch.float64, device="cuda")
        bd = torch.zeros_like(ones)
        G.gko_spmv(1.0, M, ones, 0.0, bd)
        runs = (("jacobi_mixed_f32", G.PRECOND_JACOBI, G.PRECISION_MIXED_F32),
                ("bjacobi8_mixed_f32", G.PRECOND_BLOCK_JACOBI, G.PRECISION_MIXED_F32),
                ("bjacobi8_f64", G.PRECOND_BLOCK_JACOBI, G.PRECISION_F64))
        for tag, pc, prec in runs:
            o = G.opts(precision=prec, preconditioner=pc, block_size=8)
            for rep in range(2):
                x = torch.zeros_like(ones)
                torch.cuda.synchronize()
                if rep == 1:
                    torch.cuda.nvtx.range_push("profile_solvers")
                t0 = time.perf_counter()
                r = G.gko_solve_cg(M, bd, x, 0.0, 40, o)
                torch.cuda.synchronize()
                dt = time.perf_counter() - t0
                if rep == 1:
                    torch.cuda.nvtx.range_pop()
            out[tag] = {"n": int(A.n_rows), "iterations": int(r.iterations), "ms": round(dt * 1e3, 3)}
        print(json.dumps(out))
        return
    runs = (("bicgstab", 1.0, 40, None), ("bicgstab_mixed_f32", 1.0, 40, G.PRECISION_MIXED_F32),
            ("gmres", 10.0, 30, None))
    for tag, P, iters, prec in runs:
        A = I.convdiff3d_7pt(128, P)
        M = G.from_csr(A)
        ones = torch.ones(A.n_rows, dtype=torch.float64, device="cuda")
        bd = torch.zeros_like(ones)
        G.gko_spmv(1.0, M, ones, 0.0, bd)
        fn = G.gko_solve_gmres if tag == "gmres" else G.gko_solve_bicgstab
        o = G.opts(precision=prec, inner_maxit=iters, max_outer=1) if prec is not None else None
        for rep in range(2):
            x = torch.zeros_like(ones)
            torch.cuda.synchronize()
            if rep == 1:
                torch.cuda.nvtx.range_push("profile_solvers")
            t0 = time.perf_counter()
            r = fn(M, bd, x, 0.0, iters, o) if o is not None else fn(M, bd, x, 0.0, iters)
            torch.cuda.synchronize()
            dt = time.perf_counter() - t0
            if rep == 1:
                torch.cuda.nvtx.range_pop()
        out[tag] = {"n": int(A.n_rows), "iterations": int(r.iterations), "ms": round(dt * 1e3, 3)}
        del M, A, ones, bd, x
    print(json.dumps(out))


def profile_batch(args):
    """The 4,096-system batched CG (FP64 storage, schedule 512 threads per
    block, warp threshold 0, CSR: the autotuner's choice on this workload;
    with --mixed the mixed-precision solve with reliable updates, 256 threads,
    warp threshold 64, ELL) once untimed, then once inside the NVTX range
    "profile_batch", for ncu."""
    import torch
    from paper_2006_14290_gb300 import gko as G
    from paper_2006_14290_gb300 import inputs as I

    G.load()
    sides = I.batch_sides(4096)
    systems, bs = [], []
    for i, sd in enumerate(sides):
        A, b = I.batch_system(i, int(sd))
        systems.append(A)
        bs.append(b)
    b = torch.from_numpy(np.concatenate(bs)).cuda()
    B = G.Batch(systems, storage=G.F64)
    if args.mixed:
        B.set_precision(G.PRECISION_MIXED_F32)
        B.set_schedule(64, 256, G.BATCH_ELL)
    else:
        B.set_schedule(0, 512, G.BATCH_CSR)
    out = {}
    for rep in range(2):
        x = torch.zeros(B.total_rows, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        if rep == 1:
            torch.cuda.nvtx.range_push("profile_batch")
        t0 = time.perf_counter()
        code, it, rr, st = B.cg(b, x, 1e-10, 20000)
        torch.cuda.synchronize()
        dt = time.perf_counter() - t0
        if rep == 1:
            torch.cuda.nvtx.range_pop()
        out = {"status": int(code), "iterations_total": int(it.sum()), "ms": round(dt * 1e3, 3)}
    print(json.dumps(out))


def run_ours(args):
    import torch

    rank, world, local_rank = env_rank()
    if world > 1:
        import torch.distributed as dist

        dist.init_process_group("nccl")
    torch.cuda.set_device(local_rank)
    from paper_2006_14290_gb300 import gko as G

    G.load()
    dev = torch.device("cuda", local_rank)
    stream = torch.cuda.current_stream()
    mats = workload_matrices()

    cases, skipped = build_cases(G, mats, dev)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)

    def step(events=None):
        for i, c in enumerate(cases):
            flush.fill_(float(i))
            if events is not None:
                events[i][0].record(stream)
            G.gko_spmv(1.0, c["M"], c["x"], 0.0, c["y"], stream=stream)
            if events is not None:
                events[i][1].record(stream)

    # end to end: every SpMV through the host-buffer C ABI call (x copied in
    # from pinned host memory, y copied back), cases rotating over eight
    # streams so copies overlap other cases' SpMVs (2 / 3 / 4 / 8 streams,
    # wall clock: 2.86 / 3.72 / 3.80 / 3.98 TB/s).  No L2 flush here: a case's matrix was
    # last touched 21 SpMVs (gigabytes) earlier and x arrives by copy anyway.
    E2E_STREAMS = 8
    e2e_streams = [stream] + [torch.cuda.Stream(device=dev) for _ in range(E2E_STREAMS - 1)]

    def e2e_step():
        for i, c in enumerate(cases):
            G.gko_spmv_host(1.0, c["M"], c["xh"], 0.0, c["yh"], c["x"], c["y"],
                            stream=e2e_streams[i % E2E_STREAMS])

    def barrier():
        if world > 1:
            import torch.distributed as dist
            dist.barrier()
        torch.cuda.synchronize()

    for _ in range(max(args.warmup, 3)):
        step()
    barrier()
    sampler = ClockSampler(gpu_index(local_rank))
    sampler.start()
    time.sleep(0.3)
    ev = [[[torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)] for _ in cases]
          for _ in range(args.steps)]
    t_start = torch.cuda.Event(enable_timing=True)
    t_end = torch.cuda.Event(enable_timing=True)
    barrier()
    torch.cuda.nvtx.range_push("timed_steps")
    t_start.record(stream)
    for k in range(args.steps):
        step(ev[k])
    t_end.record(stream)
    barrier()
    torch.cuda.nvtx.range_pop()
    clocks = sampler.stop()
    per_case_ms = [sum(ev[k][i][0].elapsed_time(ev[k][i][1]) for k in range(args.steps)) / args.steps
                   for i in range(len(cases))]
    kernel_ms = sum(per_case_ms)
    wall_ms = t_start.elapsed_time(t_end) / args.steps
    step_bytes = sum(c["bytes"] for c in cases)

    # end to end: host x in, host y out, through the same C ABI call
    for _ in range(max(args.warmup, 3)):
        e2e_step()
    barrier()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for st in e2e_streams[1:]:
        st.wait_event(e0)
    for _ in range(args.steps):
        e2e_step()
    for st in e2e_streams[1:]:
        stream.wait_stream(st)
    e1.record(stream)
    barrier()
    e2e_ms = e0.elapsed_time(e1) / args.steps

    kernel_ms, e2e_ms = ranks_max([kernel_ms, e2e_ms], dev)

    # formats beyond the sweep (SELL-P): same protocol, own timing loop
    extra, extra_skipped = build_cases(G, mats, dev, formats=EXTRA_FORMATS)
    for _ in range(max(args.warmup, 3)):
        for c in extra:
            G.gko_spmv(1.0, c["M"], c["x"], 0.0, c["y"], stream=stream)
    xev = [[[torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)] for _ in extra]
           for _ in range(args.steps)]
    for k in range(args.steps):
        for i, c in enumerate(extra):
            flush.fill_(float(i))
            xev[k][i][0].record(stream)
            G.gko_spmv(1.0, c["M"], c["x"], 0.0, c["y"], stream=stream)
            xev[k][i][1].record(stream)
    torch.cuda.synchronize()
    extra_ms = [sum(xev[k][i][0].elapsed_time(xev[k][i][1]) for k in range(args.steps)) / args.steps
                for i in range(len(extra))]

    peak, peak_kind = measured_peaks()
    fp64_fma = fma_peak(G, dev)
    gathers = {"f64": gather_peak(G, dev, True), "f32": gather_peak(G, dev, False)}
    dom = int(np.argmax(per_case_ms))
    dom_case = cases[dom]
    achieved = dom_case["bytes"] / (per_case_ms[dom] * 1e-3) / 1e9
    traffic = None
    tr = traffic_record()
    if tr and dom_case["label"] in tr.get("per_case_bytes", {}):
        traffic = tr["per_case_bytes"][dom_case["label"]]
    value = whole_job_gbs(world, step_bytes, kernel_ms)
    if rank == 0:
        result = {
            "metric": METRIC, "value": round(value, 2), "unit": "GB/s", "n_gpus": world, "steps": args.steps,
            "warmup": max(args.warmup, 3), "ms_per_step": round(kernel_ms, 4), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64/f32", "data": "synthetic",
            "config": {"workload": WORKLOAD, "l2": "flushed before every SpMV (256 MB write, excluded from time)",
                       "matrices": {n: {"n": int(A.n_rows), "nnz": int(A.nnz)} for n, A in mats},
                       "skipped": skipped, "frac_of_peak_value": round(value / world / peak, 4),
                       "tuned_plans": {c["label"]: c["plan"] for c in cases if c["plan"]},
                       "parallelism": f"replicas x{world}"},
            "roofline": {"bound": "hbm", "kernel": dom_case["label"], "achieved": round(achieved, 1),
                         "peak": peak, "peak_kind": peak_kind, "unit": "GB/s", "frac": round(achieved / peak, 4),
                         "traffic": traffic, "algorithmic_bytes": int(dom_case["bytes"])},
            "per_case": {c["label"]: dict({"ms": round(per_case_ms[i], 4),
                                           "GB_s": round(c["bytes"] / (per_case_ms[i] * 1e-3) / 1e9, 1),
                                           "frac": round(c["bytes"] / (per_case_ms[i] * 1e-3) / 1e9 / peak, 4)},
                                          **({"frac_fp64": round(c["nnz"] / (per_case_ms[i] * 1e-3) / fp64_fma, 4)}
                                             if c["label"].endswith("/f64") else {}),
                                          **({"frac_gather": round(c["nnz"] / (per_case_ms[i] * 1e-3)
                                                                   / gathers[c["label"][-3:]], 4)}
                                             if c["label"].startswith("powerlaw") else {}))
                         for i, c in enumerate(cases)},
            "fp64_fma_peak": {"fma_per_s": round(fp64_fma, -8), "tflops": round(2 * fp64_fma / 1e12, 3),
                              "note": "per_case frac_fp64 = nnz FMAs per SpMV / time / this rate (FP64 cases)"},
            "gather_peak": {"f64_per_s": round(gathers["f64"], -8), "f32_per_s": round(gathers["f32"], -8),
                            "note": "random gathers from an L2-resident 2^20-element vector (gko_bench_gather); "
                                    "per_case frac_gather = nnz gathers per SpMV / time / this rate "
                                    "(power-law cases: uniformly random columns)"},
            "e2e": {"value": round(whole_job_gbs(world, step_bytes, e2e_ms), 2), "unit": "GB/s",
                    "h2d_bytes_per_step": int(sum(c["x"].numel() * c["x"].element_size() for c in cases)),
                    "d2h_bytes_per_step": int(sum(c["y"].numel() * c["y"].element_size() for c in cases))},
            "extra_formats": {c["label"]: {"ms": round(extra_ms[i], 4),
                                           "GB_s": round(c["bytes"] / (extra_ms[i] * 1e-3) / 1e9, 1),
                                           "frac": round(c["bytes"] / (extra_ms[i] * 1e-3) / 1e9 / peak, 4)}
                              for i, c in enumerate(extra)},
            "extra_skipped": extra_skipped,
            "wall_ms_per_step_incl_flush": round(wall_ms, 4),
            "clocks": clocks,
            "gpu_launches": int(sum(c["launches"] for c in cases) * args.steps),
        }
        if not args.no_context:
            result["cusparse_context"] = cusparse_context(mats, dev, stream, flush, min(args.steps, 10), peak)
            result["subwarp_reduce"] = subwarp_microbench(G, dev, stream)
        if not args.no_solvers:
            oc = 0 if args.no_cpu_baseline else (os.cpu_count() or 1)
            result["solvers"] = solver_suite(G, dev, stream, flush, oracle_cores=oc)
        if not args.no_serving:
            result["serving"] = serving_suite(G)
        if world == 1 and not args.no_cpu_baseline:
            result["cpu_baseline"] = cpu_baseline(mats)
        print(json.dumps(result), file=sys.stderr, flush=True)
        print(summary_line(result), flush=True)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-solvers", action="store_true")
    ap.add_argument("--no-serving", action="store_true")
    ap.add_argument("--no-context", action="store_true", help="skip the cuSPARSE context leg")
    ap.add_argument("--profile-cases", action="store_true",
                    help="run each SpMV case once (for ncu) and print the case order")
    ap.add_argument("--small", action="store_true", help="with --profile-cases: 27-point stencil at 96^3")
    ap.add_argument("--profile-batch", action="store_true",
                    help="run the batched CG once inside an NVTX range (for ncu)")
    ap.add_argument("--mixed", action="store_true", help="with --profile-batch: the mixed-precision batched CG")
    ap.add_argument("--precond", action="store_true",
                    help="with --profile-solvers: Jacobi and block-Jacobi CG on variable coefficients 128^3")
    ap.add_argument("--profile-solvers", action="store_true",
                    help="short BiCGSTAB and GMRES(30) solves at 128^3 inside an NVTX range (for ncu)")
    args = ap.parse_args()
    if args.profile_cases:
        profile_cases(args)
        return
    if args.profile_solvers:
        profile_solvers(args)
        return
    if args.profile_batch:
        profile_batch(args)
        return
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
