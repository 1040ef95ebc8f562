#!/usr/bin/env python
"""Benchmark: IFMM factorization + preconditioned GMRES solve on one GB300.

One step = ifmm_factor (operator initialisation, leaf-to-root elimination with
colors, recompression, top-level explicit inverse) followed by bem_gmres (GMRES(30) to a true
relative residual of 1e-8, right-preconditioned by the IFMM solve, direct-sum
matvec), on the 131,072-point bumpy-sphere workload (depth 6, Chebyshev order 4,
eps = 1e-6, sigma = 3).  The tree and coloring (host, built once) and the points
and right-hand side are resident on the device before timing starts.

The JSON line reports seconds per step in the mixed-precision mode (pivots and
GMRES in FP64; Schur updates on the tensor cores as 3xTF32, recompression in
FP32; FP64-accurate float-pair matvec and FP32-stored solve) and, as "fp64", the
plain FP64 mode on the same GPU, with the error of the mixed path against it.

The timed steps run without per-launch events (launch counts only); one further
profiled step brackets every launch with CUDA events on its stream and gives the
per-class times behind "kernels" and the per-phase rooflines, whose peaks are
measured on the same GPU by the library's probes (ifmm_probe_peak) and, for HBM,
taken from MEASURED_PEAKS.json.

--rank-mode learned first trains the rank predictor on the GPU (SVD-mode ranks
of the 2,048- and 32,768-point spheres and the 65,536-point torus at eps 1e-4,
1e-6, 1e-8) and then times the learned mode; the SVD mode of the same workload
is timed beside it.

--impl reference times the CPU oracle on a bounded sample of the same workload.
With torchrun (N > 1 ranks) each rank factors and solves its own replica of the
problem (replicas only: one problem does not shard), rank 0 prints the line.
"""

from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

PEAKS_FILE = os.path.join(ROOT, "MEASURED_PEAKS.json")
METRIC = "IFMM factor+solve s at N=131k, eps=1e-6: mixed/learned vs plain FP64, same GB300"
# FP32 additions, multiplications and multiply-adds per evaluated pair of the
# float-pair direct sums: of the plain kernel for one ordered pair, of the symmetric
# one for an unordered pair, whose 1/r serves two entries (counted from the source;
# ncu's counters read 89.0, and 89.6 with the symmetric kernel's diagonal tiles)
MATVEC_DF_OPS_PER_PAIR = 89
MATVEC_SYM_OPS_PER_PAIR = 88
# FP64 operations per unordered pair of the FP64 direct sum (ncu: 13.2 with the
# diagonal tiles)
MATVEC64_OPS_PER_PAIR = 13
# BF16 MMA passes of one FP64-grade product of the level-1 inverse (digit pairs)
TOP_INVERSE_MMA_PASSES = 34
# DRAM bytes (ncu dram__bytes_read.sum + dram__bytes_write.sum) summed over the
# kernels of each class in one factor + GMRES(30) of the bumpy sphere at
# N = 32,768, depth 5, FP32 path: the --ncu-case command, captured with those
# two metrics and gpu__time_duration.sum.  ncu flushes L2 before every launch,
# so these are cold-cache bytes.  The classes listed have work linear in N at
# fixed points per leaf; the default line scales them by N / 32,768.
NCU_DRAM_BYTES_BUMPY32K = {"qr_fp32": 12.585e9, "svd_fp32": 0.411e9, "gemm_fp32": 18.609e9,
                           "gauss_jordan": 0.124e9, "solve_graph": 1.649e9}
NCU_CAPTURE_N = 32768


def max_over_ranks(value: float, dist, device) -> float:
    """The largest per-rank value (each rank times its own replica; the job takes
    as long as the slowest).  dist None: a single process."""
    if dist is None:
        return float(value)
    import torch

    t = torch.tensor([float(value)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=2)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="bumpy131k")
    ap.add_argument("--precision", default="fp32", choices=["fp32", "bf16", "fp64"])
    ap.add_argument("--rank-mode", default="svd", choices=["svd", "learned"])
    ap.add_argument("--fp64-steps", type=int, default=0, help="timed FP64 steps (0: min(steps, 4)); one warm-up")
    ap.add_argument("--sigma", type=int, default=0, help="coloring separation (0: the workload's)")
    ap.add_argument("--tau", type=int, default=2, help="levels below tau one node per color (Table 2's top level)")
    ap.add_argument("--precond", default="ifmm", choices=["ifmm", "bd"], help="IFMM factor or BD block diagonal")
    ap.add_argument("--bd-level", type=int, default=0, help="BDbot level (0: the leaf level)")
    ap.add_argument("--matvec", default="", choices=["", "df", "fp64", "fmm"],
                    help="GMRES matvec: direct sum in float pairs (default in the reduced modes) or FP64, or the "
                         "FMM representation A~ at the factor's Chebyshev order (GMRES then solves A~ x = b)")
    ap.add_argument("--wavenumber", type=float, default=0.0,
                    help="Helmholtz kernel e^{ikr}/(4 pi r) at this k (complex system, FP64 direct-sum matvec)")
    ap.add_argument("--ncu-case", action="store_true",
                    help="one factor + GMRES through the C ABI without PyTorch (for profilers); --n/--depth override "
                         "the workload's size")
    ap.add_argument("--n", type=int, default=0)
    ap.add_argument("--depth", type=int, default=0)
    ap.add_argument("--no-fp64", action="store_true", help="skip the plain FP64 comparison")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    return ap.parse_args()


class Clocks:
    """nvidia-smi samples during the timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), "--query-gpu=" + self.Q,
                                          "--format=csv,noheader,nounits", "-lms", "200"],
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
        sm, smax, reasons = [], None, set()
        names = ["active", "hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for l in self.lines:
            f = [x.strip() for x in l.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                smax = float(f[2])
            except ValueError:
                continue
            for n, v in zip(names[1:], f[5:9]):
                if v.lower() == "active":
                    reasons.add(n)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": smax, "reasons": sorted(reasons),
                "samples": len(sm)}


def sample_of(workload_name: str, factor: int):
    """A bounded sample of a workload: the same surface family, seed and
    parameters at N / factor (a power of 4) with the same mean points per leaf
    (one level less per factor 4 in N: surface-like trees grow ~4x per level)."""
    import math

    from paper_1905_10602_gb300.workloads import WORKLOADS

    w = WORKLOADS[workload_name]
    return w, w.n // factor, max(2, w.depth - int(round(math.log(factor, 4))))


def oracle_sample_seconds(workload_name: str, factor: int, repeats: int = 1):
    """The CPU oracle (as it stands) on a bounded sample of the workload, in a
    subprocess with every host core available to its BLAS; best of `repeats`."""
    code = r"""
import os, sys, time, json
sys.path.insert(0, %r)
from paper_1905_10602_gb300.workloads import WORKLOADS, surface, point_source_rhs
from oracle.ifmm import IFMMOracle
from oracle.dense import direct_matvec
from oracle.gmres import gmres
w = WORKLOADS[%r]
n, depth = %d, %d
pts = surface(w.shape, n, w.seed)
b = point_source_rhs(pts)
best = None
for _ in range(%d):
    t0 = time.perf_counter()
    o = IFMMOracle(pts, depth, w.cheb_order, w.eps, w.sigma).factor()
    x, its, rel = gmres(lambda v: direct_matvec(pts, v), b, precond=o.solve, tol=1e-8)
    t = time.perf_counter() - t0
    best = t if best is None else min(best, t)
print(json.dumps({"t": best, "n": n, "depth": depth, "its": its, "rel": rel}))
"""
    w, n_s, d_s = sample_of(workload_name, factor)
    cores = os.cpu_count() or 1
    env = dict(os.environ, OMP_NUM_THREADS=str(cores), OPENBLAS_NUM_THREADS=str(cores), MKL_NUM_THREADS=str(cores))
    out = subprocess.run([sys.executable, "-c", code % (ROOT, workload_name, n_s, d_s, repeats)], capture_output=True,
                         text=True, env=env, timeout=3600)
    if out.returncode != 0:
        raise RuntimeError(out.stderr[-2000:])
    r = json.loads(out.stdout.strip().splitlines()[-1])
    info = {"kind": "oracle", "cores": cores, "blas_threads": cores,
            "sample": f"{w.shape} N={r['n']} depth {r['depth']} (same seed, eps, order, sigma and points per leaf), "
                      f"factor + GMRES(30) to 1e-8 ({r['its']} iterations), best of {repeats}; one Python thread, "
                      f"BLAS allowed {cores} threads",
            "measured_sample_s": r["t"], "sample_n": r["n"], "sample_depth": r["depth"],
            "scaled_by": w.n / r["n"], "scaling": "work linear in N (the IFMM and its GMRES are O(N) at fixed eps "
                                                  "and points per leaf; the direct-sum matvec is not, and is a small "
                                                  "part of the oracle's time)"}
    return r["t"] * w.n / r["n"], info


def run_reference(args, rank, world):
    if rank != 0:
        return 0
    from paper_1905_10602_gb300.workloads import WORKLOADS

    times, info = [], None
    for _ in range(args.warmup):
        oracle_sample_seconds(args.workload, 64)
    for _ in range(args.steps):
        t, info = oracle_sample_seconds(args.workload, 64)
        times.append(t)
    v = sum(times) / len(times)
    w = WORKLOADS[args.workload]
    line = {"impl": "reference", "metric": METRIC, "value": v, "unit": "s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": v * 1e3, "higher_is_better": False, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": config_of(w, args.precision, args.rank_mode, world, args),
            "cpu_baseline": dict(info, value=v, unit="s"),
            "e2e": {"value": v, "unit": "s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
            "note": "each step times the oracle on the stated sample (measured_sample_s) and scales it to the "
                    "full workload's seconds (value)"}
    print(json.dumps(line), flush=True)
    return 0


def config_of(w, precision, rank_mode, world, args=None):
    sigma = (args.sigma if args is not None and args.sigma else w.sigma)
    c = {"workload": f"{w.name}: {w.shape} N={w.n}, depth {w.depth}, Chebyshev order {w.cheb_order}, "
                     f"eps {w.eps}, sigma {sigma}, GMRES(30) to 1e-8",
         "precision": precision, "rank_mode": rank_mode,
         "matvec": (args.matvec if args is not None and args.matvec else ("fp64" if precision == "fp64" else "df")),
         "global_batch": world, "l2": "working set > L2 (factor of several GB written every step)"}
    if args is not None and getattr(args, "wavenumber", 0.0):
        c["kernel"] = f"Helmholtz e^(ikr)/(4 pi r), k = {args.wavenumber}"
    if args is not None and (args.tau != 2 or args.precond != "ifmm" or args.sigma):
        c["sigma"] = sigma
        c["tau"] = args.tau
        c["precond"] = args.precond if args.precond == "ifmm" else f"BDb{args.bd_level or w.depth}"
    return c


def measured_peaks(ifmm):
    """TFLOP/s of the arithmetic units on this GPU (the library's probes) and the
    HBM copy bandwidth of MEASURED_PEAKS.json."""
    out = {k: max(ifmm.ifmm_probe_peak(k) for _ in range(2)) for k in ifmm.PEAK_KINDS}
    try:
        with open(PEAKS_FILE) as fh:
            mp = json.load(fh)
        out["hbm_gbs"] = float(mp["hbm_gbs"])
        out["hbm_source"] = "MEASURED_PEAKS.json (measured copy bandwidth)"
    except (OSError, KeyError, ValueError):
        out["hbm_gbs"] = 6800.0
        out["hbm_source"] = "fallback 6.8 TB/s (MEASURED_PEAKS.json absent)"
    out["how"] = ("ifmm_probe_peak: register-only FMA / warp-MMA chains on 8 CTAs x 256 threads per SM, best of 2, "
                  "CUDA events")
    return out


def phase_rooflines(prof, stats, peaks, precision, n, its, steps_profiled=1, matvec=None, symmetric=False):
    """One roofline entry per kernel class of the profiled step: counted work /
    CUDA-event time of the class on its launching stream, against the measured
    peak of the unit that bounds it."""
    gemm_peak = {"fp32": (peaks["tf32_mma"] / 3.0, "TF32 warp MMA peak / 3 (three MMAs per 3xTF32 product)"),
                 "bf16": (peaks["bf16_mma"], "BF16 warp MMA peak"),
                 "fp64": (peaks["fp64"], "FP64 FMA peak")}[precision]
    ents = []

    def add(kind, name, work, unit, bound, peak, peak_note):
        n_, ms = prof.get(kind, (0, 0.0))
        if not n_ or ms <= 0:
            return
        ms /= steps_profiled
        ach = work / (ms / 1e3) / (1e12 if unit == "TFLOP/s" else 1e9)
        ents.append({"phase": name, "kernel": kind, "bound": bound, "achieved": ach, "peak": peak, "unit": unit,
                     "frac": ach / peak, "ms_per_step": ms, "launches_per_step": n_ // steps_profiled,
                     "peak_note": peak_note + " (of measured)"})

    gk = "gemm_fp64" if precision == "fp64" else "gemm_fp32"
    add(gk, "a5/a7 Schur and transform GEMMs", stats.get("flops_gemm", 0.0), "TFLOP/s", "tensor" if precision != "fp64" else "alu",
        gemm_peak[0], gemm_peak[1])
    qk = "qr_fp64" if precision == "fp64" else "qr_fp32"
    add(qk, "a6 recompression pivoted QR", stats.get("flops_qr", 0.0), "TFLOP/s", "alu",
        peaks["fp64" if precision == "fp64" else "fp32"], "FP64 FMA peak" if precision == "fp64" else "FP32 FMA peak")
    sk = "svd_fp64" if precision == "fp64" else "svd_fp32"
    add(sk, "a6 recompression Jacobi SVD", stats.get("flops_svd", 0.0), "TFLOP/s", "alu",
        peaks["fp64" if precision == "fp64" else "fp32"], "FP64 FMA peak" if precision == "fp64" else "FP32 FMA peak")
    add("gauss_jordan", "a4 pivot inverses (FP64)", stats.get("flops_inv", 0.0), "TFLOP/s", "alu", peaks["fp64"], "FP64 FMA peak")
    add("gauss_jordan_big", "a9 level-1 inverse (FP64)", stats.get("flops_lu", 0.0), "TFLOP/s", "tensor",
        peaks["bf16_mma"] / TOP_INVERSE_MMA_PASSES,
        f"BF16 warp MMA peak / {TOP_INVERSE_MMA_PASSES} (passes over 8-bit digits per product)")
    apps = its + 1  # preconditioner applications per GMRES solve (one per iteration, one for x)
    add("solve_graph", "a10 IFMM solve (preconditioner)", stats.get("solve_matrix_bytes", 0.0) * apps, "GB/s", "hbm",
        peaks["hbm_gbs"], "HBM copy bandwidth")
    matvec = matvec or ("fp64" if precision == "fp64" else "df")
    if matvec == "fp64":
        add("matvec", "a11 direct-sum matvec (FP64, symmetric)", n * (n - 1) / 2.0 * (its + 1), "Gpairs/s", "alu",
            peaks["fp64"] * 1e3 / 2.0 / MATVEC64_OPS_PER_PAIR,
            f"measured FP64 FMA issue rate / {MATVEC64_OPS_PER_PAIR} FP64 operations per unordered pair")
    elif matvec == "df":
        n_, ms = prof.get("matvec", (0, 0.0))
        if n_ and ms > 0:
            ops = MATVEC_SYM_OPS_PER_PAIR if symmetric else MATVEC_DF_OPS_PER_PAIR
            per_call = float(n) * (n - 1) / 2.0 if symmetric else float(n) * n
            pairs = per_call * n_ / steps_profiled
            ach = pairs / (ms / steps_profiled / 1e3)
            pk = peaks["fp32"] * 1e12 / 2.0 / ops
            ents.append({"phase": "a11 direct-sum matvec (float pairs" + (", symmetric)" if symmetric else ")"),
                         "kernel": "matvec", "bound": "alu", "achieved": ach / 1e9, "peak": pk / 1e9,
                         "unit": "Gpairs/s", "frac": ach / pk, "ms_per_step": ms / steps_profiled,
                         "launches_per_step": n_ // steps_profiled,
                         "peak_note": f"measured FP32 FMA issue rate / {ops} FP32 operations per evaluated pair"
                                      + (" (unordered pairs: each 1/r serves two entries)" if symmetric else "")
                                      + " (of measured)"})
    return ents


def ncu_case(args):
    """One factorization + preconditioned GMRES through the C ABI, host arrays,
    no PyTorch: the command the profiles' ncu captures run."""
    from paper_1905_10602_gb300 import build as _build

    _build.build()
    from paper_1905_10602_gb300 import ifmm
    from paper_1905_10602_gb300.workloads import WORKLOADS, point_source_rhs, surface

    w = WORKLOADS[args.workload]
    n, depth = args.n or w.n, args.depth or w.depth
    pts = surface(w.shape, n, w.seed)
    b = point_source_rhs(pts)
    t = ifmm.ifmm_build_tree(pts, depth)
    ifmm.ifmm_color_levels(t, args.sigma or w.sigma, args.tau)
    arith = "fp64" if args.precision == "fp64" else "df"
    k = ifmm.default_kernel(n, arith)
    t0 = time.perf_counter()
    f = ifmm.ifmm_factor(t, w.cheb_order, w.eps, kernel=k, precision=args.precision)
    x, its, rel = ifmm.bem_gmres(t, b, precond=f, tol=1e-8, kernel=k)
    st = ifmm.ifmm_fact_stats(f)
    print(json.dumps({"case": f"{w.shape} N={n} depth {depth} {args.precision}", "seconds": time.perf_counter() - t0,
                      "gmres_iterations": its, "relres": rel, "factor_s": st["time_factor"]}), flush=True)
    return 0


def main():
    args = parse()
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if args.impl == "reference":
        return run_reference(args, rank, world)
    if args.ncu_case:
        return ncu_case(args)

    import numpy as np
    import torch

    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist

        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    from paper_1905_10602_gb300 import build as _build

    _build.build()
    from paper_1905_10602_gb300 import ifmm
    from paper_1905_10602_gb300.workloads import WORKLOADS

    if args.workload == "batch64":
        return run_batch(args, rank, world, dist, ifmm, torch)
    w = WORKLOADS[args.workload]
    pts = w.points()
    if args.wavenumber:
        from paper_1905_10602_gb300.workloads import helmholtz_source_rhs

        b_host = helmholtz_source_rhs(pts, args.wavenumber)
        args.matvec = "fp64"
        args.no_cpu = True
    else:
        b_host = w.rhs(pts)
    tree = ifmm.ifmm_build_tree(pts, w.depth)
    sigma = args.sigma or w.sigma
    ifmm.ifmm_color_levels(tree, sigma, args.tau)
    b = torch.from_numpy(b_host).cuda()
    stream = torch.cuda.current_stream()
    sptr = __import__("ctypes").c_void_p(stream.cuda_stream)
    peaks = measured_peaks(ifmm)

    def barrier():
        torch.cuda.synchronize()
        if dist is not None:
            dist.barrier()
            torch.cuda.synchronize()

    mlp, learned_info = None, None
    if args.rank_mode == "learned":
        from paper_1905_10602_gb300.learned import train_rank_model

        t0 = time.perf_counter()
        mlp, loss, nev = train_rank_model(precision="fp64" if args.precision == "fp64" else "fp32")
        learned_info = {"training_s": time.perf_counter() - t0, "training_events": nev, "final_loss": loss,
                        "trained_on": "sphere2k, sphere32k, torus65k at eps 1e-4, 1e-6, 1e-8 (SVD-mode ranks)"}

    def kernel_of(arith):
        if args.wavenumber:
            return ifmm.helmholtz_kernel(w.n, args.wavenumber)
        return ifmm.default_kernel(w.n, arith, w.cheb_order if arith == "fmm" else 0)

    def step(prec, arith, rank_mode="svd", precond=args.precond):
        k = kernel_of(arith)
        if precond == "bd":
            f = ifmm.ifmm_bd_factor(tree, args.bd_level or w.depth, kernel=k, stream=sptr)
        else:
            f = ifmm.ifmm_factor(tree, w.cheb_order, w.eps, kernel=k, precision=prec, rank_mode=rank_mode,
                                 mlp=mlp if rank_mode == "learned" else None, stream=sptr)
        x, its, rel = ifmm.bem_gmres(tree, b, precond=f, restart=30, tol=1e-8, kernel=k, stream=sptr)
        return f, its, rel, x

    def timed(prec, arith, rank_mode, steps, warmup, precond="ifmm"):
        for _ in range(warmup):
            step(prec, arith, rank_mode, precond)
        barrier()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        last = None
        for _ in range(steps):
            last = step(prec, arith, rank_mode, precond)
        e1.record(stream)
        barrier()
        return e0.elapsed_time(e1) / steps, last

    arith = args.matvec or ("fp64" if args.precision == "fp64" else "df")
    for _ in range(args.warmup):
        step(args.precision, arith, args.rank_mode)
    barrier()
    clocks = Clocks(local)
    clocks.start()
    ifmm.ifmm_profile(False)  # launch counts only inside the timed region
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    last = None
    for _ in range(args.steps):
        last = step(args.precision, arith, args.rank_mode)
    e1.record(stream)
    barrier()
    clk = clocks.stop()
    counts = ifmm.ifmm_profile_query()
    ms = e0.elapsed_time(e1) / args.steps
    ms = max_over_ranks(ms, dist, "cuda")
    fact, its, rel, x_mixed = last
    stats = ifmm.ifmm_fact_stats(fact)
    launches = counts.get("kernels", (0, 0.0))[0] // args.steps
    # one profiled step: per-launch CUDA events on the launching stream
    ifmm.ifmm_profile(True)
    pf, pits, _, _ = step(args.precision, arith, args.rank_mode)
    torch.cuda.synchronize()
    prof = ifmm.ifmm_profile_query()
    ifmm.ifmm_profile(False)
    prof.pop("kernels", None)
    pstats = ifmm.ifmm_fact_stats(pf)
    # the shared-memory, cluster and global-memory QR kernels share one work counter
    for g in ("fp32", "fp64"):
        n1, m1 = prof.get(f"qr_{g}", (0, 0.0))
        for sub in (f"qr_cluster_{g}", f"qr_global_{g}"):
            if sub in prof:
                n2, m2 = prof.pop(sub)
                n1, m1 = n1 + n2, m1 + (m2 if sub.startswith("qr_global") else 0.0)
        if n1:
            prof[f"qr_{g}"] = (n1, m1)
    tile = list(ifmm.ifmm_tree_query(tree, 0, "matvec_block"))
    phases = phase_rooflines(prof, pstats, peaks, args.precision if args.precond == "ifmm" else "fp64", w.n, pits,
                             matvec=None if args.wavenumber else arith, symmetric=len(tile) > 1 and tile[1] == 3)
    # measured DRAM traffic, where the capture applies (the default workload and path)
    captured = (args.workload == "bumpy131k" and args.precision == "fp32" and args.rank_mode == "svd"
                and args.precond == "ifmm" and arith == "df" and not args.wavenumber and args.tau == 2
                and not args.sigma)
    for e in phases:
        cap_bytes = NCU_DRAM_BYTES_BUMPY32K.get(e["kernel"]) if captured else None
        e["traffic"] = cap_bytes * w.n / NCU_CAPTURE_N if cap_bytes is not None else None
        if cap_bytes is not None:
            e["traffic_unit"] = "bytes per step (ncu, N=32,768 capture scaled by N)"
    top = max(phases, key=lambda e: e["ms_per_step"]) if phases else None
    roof = None
    if top is not None:
        roof = {"bound": top["bound"], "kernel": top["kernel"], "achieved": top["achieved"], "peak": top["peak"],
                "unit": top["unit"], "frac": top["frac"], "traffic": top.get("traffic"),
                "traffic_unit": top.get("traffic_unit"), "ms_per_step": top["ms_per_step"],
                "launches_per_step": top["launches_per_step"], "peak_note": top["peak_note"],
                "timing": "per-launch CUDA events on the launching stream, one profiled step after the timed region"}
    out = {"metric": METRIC, "value": ms / 1e3, "unit": "s", "n_gpus": world, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": False, "scaling": "weak", "vs_baseline": None,
           "dtype": "f32" if args.precision == "fp32" else ("bf16" if args.precision == "bf16" else "f64"),
           "data": "synthetic", "config": config_of(w, args.precision, args.rank_mode, world, args),
           "gmres": {"iterations": its, "relres": rel}, "factor_s": stats["time_factor"],
           "gpu_launches": int(launches),
           "kernels": {k: {"launches_per_step": n, "ms_per_step": m} for k, (n, m) in prof.items() if n},
           "roofline": roof, "phases": phases, "peaks": peaks, "clocks": clk}
    # the per-part times the measurement plan asks for, from the profiled step
    sol_n, sol_ms = prof.get("solve_graph", (0, 0.0))
    mv_n, mv_ms = prof.get("matvec", (0, 0.0))
    out["parts"] = {
        "factor_s": stats["time_factor"],
        "factor_counted_gflop": pstats.get("flops_total", 0.0) / 1e9,
        "factor_counted_gflops": pstats.get("flops_total", 0.0) / 1e9 / max(pstats.get("time_factor", 0.0), 1e-12),
        "precond_ms_per_application": sol_ms / max(pits + 1, 1) if sol_n else None,
        "matvec_ms_per_call": mv_ms / mv_n if mv_n else None,
        "gmres_iterations": its,
        "note": "counted work in the oracle's convention (2mnk per GEMM, 2n^3 per inverse, 2mn^2 - 2n^3/3 per QR, "
                "6mn^2 + 20n^3 per SVD) over the profiled step's factor time; the preconditioner and matvec times "
                "are CUDA-event times of the profiled step"}
    if learned_info is not None:
        learned_info.update({k: stats.get(k) for k in ("learned_events", "learned_sketched", "learned_fallbacks")})
        svd_ms, _ = timed(args.precision, arith, "svd", args.steps, 1)
        learned_info["svd_mode_s"] = svd_ms / 1e3
        learned_info["learned_vs_svd"] = svd_ms / ms
        out["learned"] = learned_info
    # plain FP64 on the same GPU, averaged over its own timed steps
    if not args.no_fp64 and args.precision != "fp64" and args.precond == "ifmm":
        fsteps = args.fp64_steps or min(args.steps, 4)
        f64_ms, (f64, its64, rel64, x64) = timed("fp64", "fp64", "svd", fsteps, 1)
        m_mixed = ifmm.ifmm_solve(fact, b).cpu().numpy()
        m_64 = ifmm.ifmm_solve(f64, b).cpu().numpy()
        xm, x6 = x_mixed.cpu().numpy(), x64.cpu().numpy()
        out["fp64"] = {"value": f64_ms / 1e3, "unit": "s", "steps": fsteps, "warmup": 1,
                       "gmres_iterations": its64, "relres": rel64,
                       "factor_s": ifmm.ifmm_fact_stats(f64)["time_factor"]}
        out["speedup_vs_fp64"] = (f64_ms / 1e3) / out["value"]
        out["error_vs_fp64"] = {
            "applied_inverse": float(np.linalg.norm(m_mixed - m_64) / np.linalg.norm(m_64)),
            "solution": float(np.linalg.norm(xm - x6) / np.linalg.norm(x6)),
            "note": "||M_mixed b - M_fp64 b|| / ||M_fp64 b|| for the preconditioners of the two modes, and "
                    "||x_mixed - x_fp64|| / ||x_fp64|| for the GMRES solutions (both at relative residual 1e-8)"}
    # end to end through the C ABI with host buffers: every step builds the tree
    # from pinned host points and solves from a pinned host b to a host x; one
    # untimed step first, then the same number of steps as the main timing
    if not args.no_e2e:
        pts_pin = torch.from_numpy(np.ascontiguousarray(pts)).pin_memory()
        b_pin = torch.from_numpy(np.ascontiguousarray(b_host)).pin_memory()

        def e2e_step():
            tr = ifmm.ifmm_build_tree(pts_pin, w.depth)
            ifmm.ifmm_color_levels(tr, sigma, args.tau)
            k = kernel_of(arith)
            if args.precond == "bd":
                f = ifmm.ifmm_bd_factor(tr, args.bd_level or w.depth, kernel=k)
            else:
                f = ifmm.ifmm_factor(tr, w.cheb_order, w.eps, kernel=k, precision=args.precision,
                                     rank_mode=args.rank_mode, mlp=mlp)
            xh, _, _ = ifmm.bem_gmres(tr, b_pin, precond=f, tol=1e-8, kernel=k)
            return xh

        e2e_step()
        barrier()
        t0 = time.perf_counter()
        for _ in range(args.steps):
            xh = e2e_step()
        barrier()
        te = (time.perf_counter() - t0) / args.steps
        te = max_over_ranks(te, dist, "cuda")
        n = w.n
        out["e2e"] = {"value": te, "unit": "s", "steps": args.steps,
                      "h2d_bytes_per_step": int(pts_pin.numel() * 8 + b_pin.numel() * b_pin.element_size()),
                      "d2h_bytes_per_step": int(xh.numel() * xh.element_size()),
                      "note": "per step: tree + coloring + factor + GMRES, from pinned host points and b to host x "
                              "through the public API"}
    if rank == 0 and not args.no_cpu and world == 1 and args.workload in WORKLOADS and args.precond == "ifmm":
        try:
            factor = 64 if w.n >= 65536 else 16
            val, info = oracle_sample_seconds(args.workload, factor)
            # the GPU on the very same sample, for a same-size comparison
            ws, n_s, d_s = sample_of(args.workload, factor)
            from paper_1905_10602_gb300.workloads import point_source_rhs, surface

            ps = surface(ws.shape, n_s, ws.seed)
            ts = ifmm.ifmm_build_tree(ps, d_s)
            ifmm.ifmm_color(ts, ws.sigma)
            bs = torch.from_numpy(point_source_rhs(ps)).cuda()
            ks = ifmm.default_kernel(n_s, arith)
            best = None
            for _ in range(3):
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                fs = ifmm.ifmm_factor(ts, ws.cheb_order, ws.eps, kernel=ks, precision=args.precision, stream=sptr)
                ifmm.bem_gmres(ts, bs, precond=fs, tol=1e-8, kernel=ks, stream=sptr)
                torch.cuda.synchronize()
                t = time.perf_counter() - t0
                best = t if best is None else min(best, t)
            out["cpu_baseline"] = dict(info, value=val, unit="s", gpu_same_sample_s=best,
                                       same_sample_ratio=info["measured_sample_s"] / best)
        except Exception as e:  # the oracle leg must not hide the GPU result
            out["cpu_baseline"] = {"value": None, "error": str(e)[:200]}
    if rank == 0:
        print(json.dumps(out), flush=True)
    if dist is not None:
        dist.destroy_process_group()
    return 0


def run_batch(args, rank, world, dist, ifmm, torch):
    """64 independent problems (N log-uniform in [4096, 65536], spheres / tori /
    bumpy spheres, order 4, eps 1e-6) factored and solved together per step."""
    from paper_1905_10602_gb300.workloads import batch_workloads

    ws = batch_workloads(64, 5)
    trees, bs = [], []
    for w in ws:
        pts = w.points()
        t = ifmm.ifmm_build_tree(pts, w.depth)
        ifmm.ifmm_color(t, w.sigma)
        trees.append(t)
        bs.append(w.rhs(pts))
    arith = "fp64" if args.precision == "fp64" else "df"
    ks = [ifmm.default_kernel(w.n, arith) for w in ws]

    def step():
        fs = ifmm.ifmm_factor_batched(trees, 4, 1e-6, precision=args.precision, nworkers=8, kernels=ks)
        xs, its, rel = ifmm.bem_gmres_batched(trees, bs, fs, kernels=ks, nworkers=8)
        return its, rel

    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()
    clocks = Clocks(int(os.environ.get("LOCAL_RANK", "0")))
    clocks.start()
    ifmm.ifmm_profile(False)  # launch counts only (no per-launch events)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        its, rel = step()
    torch.cuda.synchronize()
    dt = (time.perf_counter() - t0) / args.steps
    launches = ifmm.ifmm_profile_query().get("kernels", (0, 0.0))[0] // args.steps
    clk = clocks.stop()
    dt = max_over_ranks(dt, dist, "cuda")
    out = {"metric": METRIC + " (64-problem batch)", "value": dt, "unit": "s", "n_gpus": world, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": dt * 1e3, "higher_is_better": False, "scaling": "weak",
           "vs_baseline": None, "dtype": "f32" if args.precision != "fp64" else "f64", "data": "synthetic",
           "config": {"workload": "64 problems, N log-uniform in [4096, 65536], sphere/torus/bumpy, order 4, eps 1e-6, "
                                  "GMRES(30) to 1e-8, 8 worker streams", "precision": args.precision,
                      "global_batch": 64 * world},
           "problems_per_s": 64 * world / dt, "max_gmres_iterations": max(its), "max_relres": max(rel),
           "timing": "host wall clock around the batched calls (several streams)", "gpu_launches": int(launches),
           "clocks": clk}
    if rank == 0:
        print(json.dumps(out), flush=True)
    return 0


if __name__ == "__main__":
    sys.exit(main())
