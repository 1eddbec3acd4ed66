#!/usr/bin/env python
"""Benchmark: time to the k lowest eigenpairs at ||A x - lambda x||_2 <= 1e-8 on one GB300.

Workload (one "step" = one complete solve): the CI-like sparse symmetric matrix with
n = 2,000,000 rows, about 65 non-zeros per row (banded clusters of width 512 plus long-range
couplings), diagonal 0.001 i + U(0, 0.01), off-diagonals N(0, 0.005^2), seed 0; k = 16
pairs with 5 extra block vectors (the paper's choice for Full-CI runs, Sec. 4.1); initial
block = unit vectors at the 21 smallest diagonal entries.  The timed form is the mixed
precision solver (FP32 blocks and products, FP64 small matrices, FP64 refinement); the
plain FP64 solver is timed beside it.  Inputs (1.6 GB of CSR, > 1 GB of blocks) exceed the
129 MB L2, so no flush is needed between steps.

Prints one JSON line (rank 0).  `--impl reference` times the CPU FP64 oracle instead.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "time to k eigenpairs at \u2016r\u2016\u22641e-8: mixed+learned vs plain FP64 LOBPCG, 1 GB300"
N_ROWS, K, EXTRA, TOL, SEED = 2_000_000, 16, 5, 1e-8, 0
WORKLOAD = "CI-like sparse symmetric n=2,000,000, ~65 nnz/row, k=16 (+5 extra), tol 1e-8"
# Record of one complete oracle solve of this workload (iterations, wall time, threads, the
# per-iteration time of its first iterations), written by oracle/record_full_solve.py, which
# calls only the oracle.  Both CPU legs scale it to the machine's cores.
ORACLE_RECORD = os.path.join(ROOT, "oracle", "records", "ci2m_seed0.json")
FP64_PEAK_SOURCE = "FP64 FMA rate measured in this run (lobpcg_probe_fma_rate)"
DIGIT_PRODUCTS = 34  # FP16 products of one FP64 multiply-add (csrc/slices.cuh)
DF_OPS_PER_TERM = 15  # FP32 operations of one double-float multiply-add (dfloat.cuh df_fma)


def log(*a):
    print(*a, file=sys.stderr, flush=True)


def dist_env():
    return int(os.environ.get("RANK", 0)), int(os.environ.get("WORLD_SIZE", 1)), int(os.environ.get("LOCAL_RANK", 0))


def max_over_ranks(x: float, world: int, device: str = "cuda") -> float:
    """The largest x over the ranks of the default process group (x itself for one rank):
    the bench's time is the slowest replica's."""
    if world <= 1:
        return x
    import torch
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def make_problem(n_rows=N_ROWS):
    import synth
    cache = f"/tmp/lobpcg_bench_ci_{n_rows}_{SEED}.npz"
    if os.path.exists(cache):
        z = np.load(cache)
        a = synth.CSR(n=int(z["n"]), row_ptr=z["row_ptr"], col_idx=z["col_idx"], val=z["val"], diag=z["diag"])
    else:
        a = synth.sparse_ci(n=n_rows, seed=SEED)
        try:
            np.savez(cache, n=a.n, row_ptr=a.row_ptr, col_idx=a.col_idx, val=a.val, diag=a.diag)
        except OSError:
            pass
    x0 = synth.diag_guess(a.diag, K + EXTRA, seed=SEED, noise=0.0)
    return a, x0


class Clocks:
    """nvidia-smi sampling of SM clocks and throttle reasons during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu: int):
        self.gpu = gpu
        self.proc = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
        return self

    def __exit__(self, *exc):
        self.out = ""
        if self.proc:
            self.proc.terminate()
            try:
                self.out, _ = self.proc.communicate(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
                self.out, _ = self.proc.communicate()

    def summary(self):
        sm, mx, reasons = [], 0.0, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in (self.out or "").splitlines():
            f = [x.strip() for x in line.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx = max(mx, float(f[2]))
            except ValueError:
                continue
            for nm, v in zip(names, f[5:9]):
                if v.lower().startswith("active") or v == "0x1":
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": mx or None,
                "reasons": sorted(reasons), "samples": len(sm)}


def measured_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            p = json.load(f)
        return float(p["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


def tensor_peak():
    """Dense FP16 / BF16 tensor rate in TFLOP/s and its source."""
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return float(json.load(f)["bf16_tflops"]), "measured (cuBLAS bf16, burst)"
    except Exception:
        return 1900.0, "fallback (cuBLAS bf16, burst)"


def mean_offdiag_row_norm(a):
    """c = mean over rows of the off-diagonal row 2-norm (the learned preconditioner's
    scale; the damped diagonal floors |d_i - theta| at it)."""
    rows = np.repeat(np.arange(a.n), np.diff(a.row_ptr))
    off = a.col_idx != rows
    return float(np.mean(np.sqrt(np.bincount(rows[off], weights=a.val[off] ** 2, minlength=a.n))))


def oracle_sample(a, x0):
    """Bounded sample of the oracle, as it stands, on the full workload: its initialisation
    alone, then the initialisation plus two iterations (about 10 s of CPU work)."""
    import oracle
    oracle.lib()
    t0 = time.perf_counter()
    oracle.lobpcg(a, a.diag, K, x0, extra=EXTRA, tol=TOL, maxiter=0, hist_cap=2)
    t1 = time.perf_counter()
    oracle.lobpcg(a, a.diag, K, x0, extra=EXTRA, tol=TOL, maxiter=2, hist_cap=4)
    t2 = time.perf_counter()
    init = t1 - t0
    per_it = max((t2 - t1) - init, 1e-9) / 2.0
    return init, per_it, t2 - t0


def oracle_time_to_solution(a, x0):
    """The one formula of both CPU legs: the oracle's time to the k pairs on this machine.

    A complete oracle solve of the workload is too long for a benchmark run, so it is
    extrapolated from a measured sample.  With the record of a complete oracle solve (its
    wall time T_rec and the per-iteration time p_rec of its first iterations, on the cores
    where it ran), the estimate is T_rec * p / p_rec, p the per-iteration time measured
    here: the record carries the oracle's own iteration count and the shrinking active
    block of soft locking.  Without a record: init + iterations x p at the full width."""
    import oracle
    init, per_it, spent = oracle_sample(a, x0)
    cores = oracle.threads()
    rec = None
    try:
        with open(ORACLE_RECORD) as f:
            rec = json.load(f)
    except (OSError, ValueError):
        rec = None
    if rec and rec.get("status") == 0:
        value = rec["seconds"] * per_it / rec["per_iteration_seconds"]
        sample = (f"extrapolated: oracle init + 2 iterations on the full n={N_ROWS} workload here ({spent:.1f} s of "
                  f"CPU work, {per_it:.2f} s per iteration on {cores} threads) scaled by the record of a complete "
                  f"oracle solve ({rec['iterations']} iterations, {rec['seconds']:.0f} s on {rec['threads']} "
                  f"threads at {rec['per_iteration_seconds']:.2f} s per early iteration)")
    else:
        value = None
        sample = f"no complete oracle solve on record; sample {spent:.1f} s, {per_it:.2f} s per iteration"
    return {"value": value, "unit": "s", "cores": cores, "kind": "oracle", "extrapolated": True, "sample": sample,
            "init_seconds": init, "per_iteration_seconds": per_it}


def run_reference(args):
    rank, world, _ = dist_env()
    if rank != 0:
        return 0
    a, x0 = make_problem()
    samples = []
    est = None
    for step in range(args.warmup + args.steps):
        t0 = time.perf_counter()
        est = oracle_time_to_solution(a, x0)
        if step >= args.warmup:
            samples.append((time.perf_counter() - t0, est))
    per_step = statistics.median(t for t, _ in samples)
    value = statistics.median(e["value"] for _, e in samples if e["value"] is not None) if est["value"] else None
    if value is None:
        print(json.dumps({"impl": "reference", "unavailable": "no complete oracle solve on record to scale"}))
        return 0
    base = dict(samples[-1][1])
    base["value"] = value
    line = {"metric": METRIC, "value": value, "unit": "s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": per_step * 1e3, "higher_is_better": False, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic", "impl": "reference",
            "config": {"workload": WORKLOAD, "l2": "inputs larger than L2"},
            "cpu_baseline": base,
            "e2e": {"value": value, "unit": "s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


def run_ours(args):
    import torch
    rank, world, local = dist_env()
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    torch.cuda.set_device(local)
    import __graft_entry__
    __graft_entry__.build()
    import paper_2305_06668_gb300 as lb

    # FMA-pipe peaks of this GPU, measured now (denominators of the "alu" rooflines)
    fp64_peak = lb.probe_fma_rate(fp64=True)
    fp32_peak = lb.probe_fma_rate(fp64=False)
    a, x0_np = make_problem(args.n)
    t = lb.upload_csr(a)
    x0 = torch.from_numpy(x0_np).cuda()
    stream = torch.cuda.current_stream()
    weights = lb.load_mlp_weights()
    mixed = lb.Solver(**t, extra=EXTRA, precision=lb.MIXED, precond=lb.PREC_LEARNED, mlp_weights=weights,
                      profile=True, maxiter=args.maxiter)
    for _ in range(args.warmup):
        r = mixed.solve(K, TOL, X0=x0)
    torch.cuda.synchronize()

    def barrier():
        if world > 1:
            torch.distributed.barrier()
        torch.cuda.synchronize()

    infos = []
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with Clocks(local) as clk:
        barrier()
        ev0.record(stream)
        for _ in range(args.steps):
            r = mixed.solve(K, TOL, X0=x0)
            infos.append((r.status, r.info, r.resnorms.max(), r.evals.copy()))
        ev1.record(stream)
        barrier()
    total = max_over_ranks(ev0.elapsed_time(ev1) / 1e3, world)
    per_solve = total / args.steps
    statuses = [s for s, *_ in infos]
    last = infos[-1][1]

    if args.profile:
        # profiling run (ncu): the timed solves only
        mixed.close()
        if rank == 0:
            print(json.dumps({"profile_run": True, "n": a.n, "s_per_solve": per_solve,
                              "iterations": last["iterations"], "status": [lb.STATUS_NAMES[s] for s in statuses]}))
        return 0
    # the comparison the metric names: plain FP64 GPU solves of the same problem (median of
    # args.fp64_runs; the iteration count of FP64 LOBPCG on this matrix moves a lot with
    # rounding), and the ablations that split the gain into its precision and
    # preconditioner parts: FP64 + learned, mixed + diagonal, and mixed + damped diagonal
    # (the classical control for the learned preconditioner)
    def timed_solve(**kw):
        s = lb.Solver(**t, extra=EXTRA, maxiter=args.maxiter, **kw)
        rr = s.solve(K, TOL, X0=x0)
        s.close()
        return rr
    plain = [timed_solve(precision=lb.FP64) for _ in range(args.fp64_runs)]
    r64 = sorted(plain, key=lambda rr: rr.info["seconds"])[len(plain) // 2]
    fp64_time = r64.info["seconds"]
    ablations = {}
    c_rho = mean_offdiag_row_norm(a)  # the damped diagonal's floor: the learned model's own scale
    for name, kw in (("fp64_learned", dict(precision=lb.FP64, precond=lb.PREC_LEARNED, mlp_weights=weights)),
                     ("mixed_diagonal", dict(precision=lb.MIXED)),
                     ("mixed_damped_diagonal", dict(precision=lb.MIXED, precond_floor=c_rho))):
        rr = timed_solve(**kw)
        ablations[name] = {"seconds": rr.info["seconds"], "iterations": rr.info["iterations"],
                           "fp64_iterations": rr.info["fp64_iterations"], "status": lb.STATUS_NAMES[rr.status],
                           "max_resnorm": float(np.max(rr.resnorms)),
                           "eig_max_rel_diff_vs_fp64": float(np.max(np.abs(rr.evals - r64.evals) /
                                                                    np.maximum(1, np.abs(r64.evals))))}

    # rooflines of the main kernels from the phase timings of the timed solves (CUDA
    # events on the solver stream); the dominant phase's is reported as "roofline"
    hbm_peak, peak_kind = measured_peaks()
    tot = lambda key, ph: sum(i[key][ph] for _, i, _, _ in infos)
    ph_all = {ph: tot("phase_seconds", ph) for ph in lb.PHASES}
    ph64 = {ph: tot("phase_seconds_fp64", ph) for ph in lb.PHASES}
    nnz, n = a.nnz, a.n
    l32 = sum(i["spmm_launches"] - i["spmm_launches_fp64"] for _, i, _, _ in infos)
    c32 = sum(i["spmm_columns"] - i["spmm_columns_fp64"] for _, i, _, _ in infos)
    l64 = sum(i["spmm_launches_fp64"] for _, i, _, _ in infos)
    c64 = sum(i["spmm_columns_fp64"] for _, i, _, _ in infos)
    rooflines = {}
    if l32:
        t32 = (ph_all["spmm"] - ph64["spmm"]) / l32
        cols = c32 / l32
        # algorithmic bytes of one FP32 product: values + column indices + row pointers + read W + write AW
        b32 = nnz * (4 + 4) + (n + 1) * 8 + 2 * n * cols * 4
        rooflines["spmm_fp32"] = {"kernel": "spmm_band_packed_kernel + spmm_csr_add_kernel (A W, FP32, band / "
                                            "long-range split)", "bound": "hbm",
                                  "achieved": b32 / t32 / 1e9, "peak": hbm_peak, "unit": "GB/s",
                                  "frac": b32 / t32 / 1e9 / hbm_peak, "traffic": None,
                                  "bytes_per_launch": b32, "avg_launch_s": t32, "peak_source": peak_kind}
    df = bool(infos[-1][1]["df_products"])
    if l64:
        t64 = ph64["spmm"] / l64
        cols = c64 / l64
        f64 = 2.0 * nnz * cols
        if df:
            # double-float product on the FP32 pipes (the block's split into float pairs included)
            ops = f64 / 2.0 * DF_OPS_PER_TERM
            rooflines["spmm_fp64"] = {"kernel": "spmm_csr_df_kernel (A W, FP64 refinement in double-float on the "
                                                "FP32 pipes, row-parallel)", "bound": "alu",
                                      "achieved": ops / t64 / 1e12, "peak": fp32_peak / 2, "unit": "TFLOP/s",
                                      "frac": ops / t64 / 1e12 / (fp32_peak / 2),
                                      "ops": "FP32 pipe operations, 15 per FP64-equivalent multiply-add",
                                      "fp64_equivalent_tflops": f64 / t64 / 1e12, "traffic": None,
                                      "flops_per_launch": ops, "avg_launch_s": t64,
                                      "peak_source": "FP32 FMA instruction rate measured in this run "
                                                     "(lobpcg_probe_fma_rate / 2)"}
        else:
            rooflines["spmm_fp64"] = {"kernel": "spmm_csr_add_kernel<double> (A W, FP64 refinement, row-parallel)",
                                      "bound": "alu",
                                      "achieved": f64 / t64 / 1e12, "peak": fp64_peak, "unit": "TFLOP/s",
                                      "frac": f64 / t64 / 1e12 / fp64_peak, "traffic": None,
                                      "flops_per_launch": f64, "avg_launch_s": t64,
                                      "peak_source": FP64_PEAK_SOURCE}
    # the FP64 block updates of the refinement, timed per launch with CUDA events: digit products above
    # their size rules (34 FP16 products per FP64 multiply-add, of the padded 32 columns only the used ones
    # counted), the double-float or FMA kernels below, each against its own peak
    def total(key):
        return sum(i[key] for _, i, _, _ in infos)
    dt_, df_, dl_ = total("update_digit_seconds"), total("update_digit_flops"), total("update_digit_launches")
    ot, of, ol = (total("update_fp64_seconds") - dt_, total("update_fp64_flops") - df_,
                  total("update_fp64_launches") - dl_)
    if dl_ and dt_ > 0:
        peak, source = tensor_peak()
        ops = df_ * DIGIT_PRODUCTS
        rooflines["update_fp64"] = {"kernel": "update64_kernel (FP64 block updates through FP16 digit products, "
                                              "tcgen05: X = V u_x, P = V u_p, W -= Y C, W <- W T)",
                                    "bound": "alu",
                                    "limited_by": "integer pipe (cutting into digits, joining of the sums)",
                                    "achieved": ops / dt_ / 1e12, "peak": peak, "unit": "TFLOP/s",
                                    "frac": ops / dt_ / 1e12 / peak,
                                    "ops": "FP16 tensor flops, 34 digit products per FP64 multiply-add",
                                    "fp64_equivalent_tflops": df_ / dt_ / 1e12, "traffic": None,
                                    "launches": dl_, "flops_per_launch": ops / dl_, "avg_launch_s": dt_ / dl_,
                                    "peak_source": source}
    if ol and ot > 0:
        ops = of / 2.0 * DF_OPS_PER_TERM if df else of
        rooflines["update_fp64_small"] = {
            "kernel": ("update_df_async_kernel (FP64 block updates below the size rule, double-float)" if df
                       else "update_kernel<double> (FP64 block updates below the size rule)"),
            "bound": "alu", "achieved": ops / ot / 1e12, "peak": fp32_peak / 2 if df else fp64_peak,
            "unit": "TFLOP/s", "frac": ops / ot / 1e12 / (fp32_peak / 2 if df else fp64_peak),
            "fp64_equivalent_tflops": of / ot / 1e12, "traffic": None, "launches": ol,
            "flops_per_launch": ops / ol, "avg_launch_s": ot / ol,
            "peak_source": ("FP32 FMA instruction rate measured in this run (lobpcg_probe_fma_rate / 2)" if df
                            else FP64_PEAK_SOURCE)}
    # the FP32 Rayleigh-Ritz Grams (tcgen05 kernel): algorithmic bytes 2 n s 4 per Gram over the
    # FP32 part of the Rayleigh-Ritz Gram phase
    gb = sum(i["rr_gram32_bytes"] for _, i, _, _ in infos)
    gc = sum(i["rr_gram32_count"] for _, i, _, _ in infos)
    gt = ph_all["rr_gram"] - ph64["rr_gram"]
    if gc and gt > 0:
        rooflines["gram_fp32"] = {"kernel": "gram_umma_kernel + reduce (V^T AV, FP32, tcgen05 3xTF32)",
                                  "bound": "hbm", "achieved": gb / gt / 1e9, "peak": hbm_peak, "unit": "GB/s",
                                  "frac": gb / gt / 1e9 / hbm_peak, "traffic": None, "bytes_per_launch": gb / gc,
                                  "avg_launch_s": gt / gc, "peak_source": peak_kind}
    share = {k: v / max(sum(ph_all.values()), 1e-30) for k, v in ph_all.items()}
    roofline = dict(rooflines.get("update_fp64", rooflines.get("spmm_fp32", {})))
    roofline["phase_share"] = share
    roofline["dominant_phase"] = max(share, key=share.get)
    # end to end through the C ABI from pinned host buffers: H2D of the matrix and the
    # initial block, context creation, solve, D2H of the eigenvectors
    host = {k: v.cpu().pin_memory() for k, v in t.items()}
    hx0 = x0.cpu().pin_memory()
    e2e_times = []
    h2d = sum(v.numel() * v.element_size() for v in host.values()) + hx0.numel() * 8
    d2h = n * K * 8
    for _ in range(max(1, min(2, args.steps))):
        torch.cuda.synchronize()
        e0 = time.perf_counter()
        dt = {k: v.to("cuda", non_blocking=True) for k, v in host.items()}
        dx0 = hx0.to("cuda", non_blocking=True)
        s = lb.Solver(**dt, extra=EXTRA, precision=lb.MIXED, precond=lb.PREC_LEARNED, mlp_weights=weights,
                      maxiter=args.maxiter)
        rr = s.solve(K, TOL, X0=dx0)
        ev = rr.evecs.cpu()
        s.close()
        torch.cuda.synchronize()
        e2e_times.append(time.perf_counter() - e0)
        del dt, dx0, ev

    base = None
    if rank == 0 and world == 1 and not args.no_cpu:
        base = oracle_time_to_solution(a, x0_np)
    mixed.close()
    if rank != 0:
        return 0
    summary = clk.summary()
    line = {"metric": METRIC, "value": per_solve, "unit": "s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": per_solve * 1e3, "higher_is_better": False, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32+f64", "data": "synthetic",
            "config": {"workload": WORKLOAD, "form": "mixed precision (FP32 blocks, FP64 small matrices) + FP64 "
                       "refinement, learned preconditioner (trained weights shipped with the package)",
                       "l2": "inputs larger than L2 (no flush needed)",
                       "parallelism": f"replicas x{world}" if world > 1 else "1 GPU"},
            "status": [lb.STATUS_NAMES[s] for s in statuses],
            "iterations": last["iterations"], "fp64_iterations": last["fp64_iterations"],
            "max_resnorm": float(infos[-1][2]),
            "fp64_seconds": fp64_time, "fp64_iterations_plain": r64.info["iterations"],
            "fp64_runs": [{"seconds": rr.info["seconds"], "iterations": rr.info["iterations"],
                           "status": lb.STATUS_NAMES[rr.status]} for rr in plain],
            "fp64_status": lb.STATUS_NAMES[r64.status], "speedup_vs_fp64": fp64_time / per_solve,
            "ablations": ablations,
            "peaks": {"hbm_gbs": hbm_peak, "hbm_source": peak_kind, "fp64_tflops": fp64_peak,
                      "fp32_tflops": fp32_peak, "fma_source": "lobpcg_probe_fma_rate in this run"},
            "precond_fallback": last["precond_fallback"],
            "eig_max_rel_diff_vs_fp64": float(np.max(np.abs(infos[-1][3] - r64.evals) / np.maximum(1, np.abs(r64.evals)))),
            "phase_seconds_per_solve": {k: v / args.steps for k, v in ph_all.items()},
            "phase_seconds_fp64_per_solve": {k: v / args.steps for k, v in ph64.items()},
            "roofline": roofline, "rooflines": rooflines, "clocks": summary,
            "e2e": {"value": min(e2e_times), "unit": "s", "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(d2h)},
            "gpu_launches": int(sum(i["kernel_launches"] for _, i, _, _ in infos))}
    if base:
        line["cpu_baseline"] = base
    print(json.dumps(line), flush=True)
    if world > 1:
        torch.distributed.destroy_process_group()
    return 0


def run_batched(args):
    """The batched serving workload (a separate line, not the headline): 256 problems of the
    cfg1 construction, n ~ U[10,000, 500,000], k ~ U{1..32}, generated on the GPU; all
    solved with lobpcg_solve_batched (mixed precision + FP64 refinement, one stream per
    problem) against the same problems solved one by one with the plain FP64 path."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2305_06668_gb300 as lb
    import synth
    specs = synth.batched_specs(args.nprob, seed=0)
    mats, x0s = [], []
    for n, k, sd in specs:
        t = synth.sparse_cfg1_torch(n, sd)
        mats.append(t)
        x0s.append(synth.diag_guess_torch(t["diag"], k))
    torch.cuda.synchronize()
    ks = [k for _, k, _ in specs]
    streams = [torch.cuda.Stream() for _ in specs]
    # serving-style contexts: created once, the product kernels autotuned on the first
    # (warm-up) solve and reused by the timed ones
    batched = [lb.Solver(**t, precision=lb.MIXED, autotune=True, stream=st) for t, st in zip(mats, streams)]
    times = []
    for rep in range(args.warmup + args.steps):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        rb = lb.solve_batched(batched, ks, [TOL] * len(ks), x0s, nthreads=args.threads)
        torch.cuda.synchronize()
        if rep >= args.warmup:
            times.append(time.perf_counter() - t0)
    torch.cuda.synchronize()
    # one by one with the plain FP64 path: context creation, solve, release per problem
    seq = 0.0
    r1 = []
    for t, k, x in zip(mats, ks, x0s):
        s = lb.Solver(**t, precision=lb.FP64)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        r1.append(s.solve(k, TOL, X0=x))
        torch.cuda.synchronize()
        seq += time.perf_counter() - t0
        s.close()
    diff = max(float(np.max(np.abs(a.evals - b.evals) / np.maximum(1, np.abs(b.evals)))) for a, b in zip(rb, r1))
    line = {"metric": "time to solve 256 independent problems at \u2016r\u2016\u22641e-8 (batched)",
            "value": min(times), "unit": "s", "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
            "higher_is_better": False, "dtype": "f32+f64", "data": "synthetic",
            "config": {"workload": f"{len(specs)} cfg1-recipe problems, n ~ U[10k, 500k], k ~ U{{1..32}}",
                       "sum_n": int(sum(n for n, _, _ in specs)), "sum_nnz": int(sum(int(t['row_ptr'][-1]) for t in mats)),
                       "form": "lobpcg_solve_batched, mixed precision + FP64 refinement, one stream per problem"},
            "sequential_plain_fp64_s": seq, "speedup_vs_sequential_fp64": seq / min(times),
            "status_ok": sum(r.status == lb.OK for r in rb), "max_rel_eig_diff_vs_fp64": diff,
            "iterations_total": int(sum(r.info["iterations"] for r in rb))}
    print(json.dumps(line), flush=True)
    return 0


def run_small_config(args):
    """A side line per further configuration (not the headline): cfg1, the n = 4096 sparse
    problem (k = 4, unit vectors plus N(0, 1e-3) noise), or the dense CASSCF-like problem
    (n = 8192, rank 256, k = 8).  Each form is solved best-of-`steps` after `warmup` solves:
    mixed + learned, plain FP64, and the two ablations; the dense product's bandwidth is
    measured from the profiled phase timings."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2305_06668_gb300 as lb
    import synth
    weights = lb.load_mlp_weights()
    if args.config == "cfg1":
        a = synth.sparse_cfg1(n=4096, seed=0)
        t = lb.upload_csr(a)
        x0 = torch.from_numpy(synth.diag_guess(a.diag, 4, seed=0)).cuda()
        k, name = 4, "cfg1: sparse n=4096, 16 couplings per row mirrored, k=4, X0 unit vectors + N(0,1e-3)"
        mat = t
        nbytes64 = None
    else:
        A, d = synth.dense_casscf(n=8192, seed=0, rank=256)
        mat = dict(diag=torch.from_numpy(d).cuda(), dense=torch.from_numpy(A).cuda())
        x0 = torch.from_numpy(synth.diag_guess(d, 8, seed=0)).cuda()
        k, name = 8, "dense CASSCF-like: n=8192, A = D + U S U^T rank 256, k=8, X0 unit vectors + N(0,1e-3)"
        nbytes64 = 8192 * 8192 * 8
    forms = {"mixed_learned": dict(precision=lb.MIXED, precond=lb.PREC_LEARNED, mlp_weights=weights),
             "fp64": dict(precision=lb.FP64),
             "fp64_learned": dict(precision=lb.FP64, precond=lb.PREC_LEARNED, mlp_weights=weights),
             "mixed_diagonal": dict(precision=lb.MIXED)}
    out = {}
    for fname, kw in forms.items():
        s = lb.Solver(**mat, maxiter=3000, profile=True, **kw)
        for _ in range(args.warmup):
            s.solve(k, TOL, X0=x0)
        best = None
        for _ in range(max(1, args.steps)):
            r = s.solve(k, TOL, X0=x0)
            if best is None or r.info["seconds"] < best.info["seconds"]:
                best = r
        s.close()
        i = best.info
        row = {"seconds": i["seconds"], "iterations": i["iterations"], "fp64_iterations": i["fp64_iterations"],
               "status": lb.STATUS_NAMES[best.status], "max_resnorm": float(np.max(best.resnorms)),
               "evals": [float(v) for v in best.evals]}
        if nbytes64:
            # dense products: FP64 (n^2 * 8 B of A) in the FP64 phase, FP32 (n^2 * 4 B) in the FP32 one
            l64, l32 = i["spmm_launches_fp64"], i["spmm_launches"] - i["spmm_launches_fp64"]
            t64 = i["phase_seconds_fp64"]["spmm"]
            t32 = i["phase_seconds"]["spmm"] - t64
            if l64:
                row["dense_product_fp64_gbs"] = nbytes64 * l64 / t64 / 1e9
            if l32:
                row["dense_product_fp32_gbs"] = nbytes64 / 2 * l32 / t32 / 1e9
        out[fname] = row
    ref = out["fp64"]["evals"]
    for row in out.values():
        row["eig_max_rel_diff_vs_fp64"] = float(np.max(np.abs(np.array(row["evals"]) - ref) /
                                                    np.maximum(1, np.abs(ref))))
    hbm, _ = measured_peaks()
    line = {"metric": METRIC, "value": out["mixed_learned"]["seconds"], "unit": "s", "n_gpus": 1,
            "steps": args.steps, "warmup": args.warmup, "higher_is_better": False, "dtype": "f32+f64",
            "data": "synthetic", "config": {"workload": name, "form": "mixed + learned (best of steps)"},
            "fp64_seconds": out["fp64"]["seconds"],
            "speedup_vs_fp64": out["fp64"]["seconds"] / out["mixed_learned"]["seconds"], "forms": out,
            "hbm_peak_gbs": hbm}
    print(json.dumps(line), flush=True)
    return 0


def run_gram_config(args):
    """Side line: the FP32 Gram C = X^T Y at n = 2*10^6 rows, tcgen05 kernel against the
    warp-level mma.sync kernel, on the Gram shapes of the headline solve (63 x 63 and 42 x 21
    over two blocks, X^T X over 21 columns) and the widest block (96 x 96).  Each call is timed
    with CUDA events around the C-ABI call, which includes its scratch set-up; the kernels'
    own times come from an ncu launch list of this command."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2305_06668_gb300 as lb
    n = N_ROWS
    g = torch.Generator(device="cuda").manual_seed(SEED)
    shapes = [("63x63", 63, 63, 64, False), ("42x21", 42, 21, 44, False), ("21x21_same", 21, 21, 24, True),
              ("96x96", 96, 96, 96, False)]
    out = {}
    for name, p, q, ld, same in shapes:
        X = torch.randn(n, ld, device="cuda", generator=g)[:, :p]
        Y = X[:, :q] if same else torch.randn(n, ld, device="cuda", generator=g)[:, :q]
        nbytes = n * (p + (0 if same else q)) * 4
        row = {}
        for kname, fn in (("tcgen05", lb.gram_f32_tcgen05), ("mma_sync", lb.gram_f32)):
            for _ in range(args.warmup):
                fn(X, Y)
            ts = []
            for _ in range(max(1, args.steps)):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record()
                fn(X, Y)
                e1.record()
                torch.cuda.synchronize()
                ts.append(e0.elapsed_time(e1) * 1e-3)
            row[kname] = {"call_seconds": float(np.median(ts))}
        row["bytes"] = nbytes
        out[name] = row
        del X, Y
    print(json.dumps({"side_line": "fp32 gram kernels", "n": n, "shapes": out}), flush=True)
    return 0


def run_damping_config(args):
    """Side line: the learned preconditioner against damped diagonal ones, a classical
    control.  Held-out CI-like matrices (n = 100,000, seeds 2100-2102, not used in
    training), k = 16 (+5 extra), tol 1e-8, FP64: the diagonal preconditioner with its
    denominator floored at alpha * c for several alpha (c = mean off-diagonal row 2-norm, the
    learned preconditioner's own scale), and the learned one."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2305_06668_gb300 as lb
    import synth
    w = lb.load_mlp_weights()
    alphas = (0.0, 0.25, 1.0, 4.0, 16.0)
    out = []
    for seed in (2100, 2101, 2102):
        a = synth.sparse_ci(n=100_000, seed=seed)
        c = mean_offdiag_row_norm(a)
        t = lb.upload_csr(a)
        x0 = torch.from_numpy(synth.diag_guess(a.diag, K + EXTRA, seed=seed, noise=0.0)).cuda()
        forms = [(f"diag_floor_{al:g}c", dict(precond_floor=al * c)) for al in alphas]
        forms.append(("learned", dict(precond=lb.PREC_LEARNED, mlp_weights=w)))
        for name, kw in forms:
            s = lb.Solver(**t, extra=EXTRA, maxiter=20000, **kw)
            r = s.solve(K, TOL, X0=x0)
            s.close()
            out.append({"seed": seed, "form": name, "c": c, "status": lb.STATUS_NAMES[r.status],
                        "iterations": r.info["iterations"], "seconds": r.info["seconds"],
                        "max_resnorm": float(np.max(r.resnorms)), "evals0": float(r.evals[0])})
            log(json.dumps(out[-1]))
    print(json.dumps({"side_line": "learned vs damped diagonal preconditioners (FP64, held-out seeds)",
                      "n": 100000, "runs": out}), flush=True)
    return 0


def run_precond_config(args):
    """Side line in the manner of the paper's Table 1 (Sec. 4.4): iterations and time of
    LOBPCG with the diagonal, tridiagonal and learned preconditioners, FP64, tol 1e-8, on
    cfg1 (n = 4096, k = 4), the dense CASSCF-like matrix (n = 8192, k = 8) and a held-out
    CI-like matrix (n = 100,000, seed 2100, k = 16 + 5).  Each form: one warm-up solve, then
    the best of `steps`; the preconditioner's own time per iteration from the profiled
    phase timings."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2305_06668_gb300 as lb
    import synth
    w = lb.load_mlp_weights()
    cases = []
    a = synth.sparse_cfg1(n=4096, seed=0)
    cases.append(("cfg1 n=4096 k=4", lb.upload_csr(a), synth.diag_guess(a.diag, 4, seed=0), 4, 0))
    A, d = synth.dense_casscf(n=8192, seed=0, rank=256)
    cases.append(("dense CASSCF-like n=8192 k=8", dict(diag=torch.from_numpy(d).cuda(), dense=torch.from_numpy(A).cuda()),
                  synth.diag_guess(d, 8, seed=0), 8, 0))
    c = synth.sparse_ci(n=100_000, seed=2100)
    cases.append(("CI-like n=100000 seed 2100 k=16+5", lb.upload_csr(c),
                  synth.diag_guess(c.diag, K + EXTRA, seed=2100, noise=0.0), K, EXTRA))
    forms = (("diagonal", dict(precond=lb.PREC_DIAG)), ("tridiagonal", dict(precond=lb.PREC_TRIDIAG)),
             ("learned", dict(precond=lb.PREC_LEARNED, mlp_weights=w)))
    out = []
    for name, mat, x0np, k, extra in cases:
        x0 = torch.from_numpy(x0np).cuda()
        for fname, kw in forms:
            s = lb.Solver(**mat, extra=extra, maxiter=20000, profile=True, **kw)
            s.solve(k, TOL, X0=x0)
            best = None
            for _ in range(max(1, args.steps)):
                r = s.solve(k, TOL, X0=x0)
                if best is None or r.info["seconds"] < best.info["seconds"]:
                    best = r
            s.close()
            i = best.info
            ph = i["phase_seconds"]
            out.append({"case": name, "preconditioner": fname, "status": lb.STATUS_NAMES[best.status],
                        "iterations": i["iterations"], "seconds": i["seconds"],
                        "precond_ms_per_iteration": 1e3 * ph["precond"] / max(1, i["iterations"] + 1),
                        "max_resnorm": float(np.max(best.resnorms)), "evals0": float(best.evals[0])})
            log(json.dumps(out[-1]))
    print(json.dumps({"side_line": "preconditioners as in Table 1: diagonal, tridiagonal, learned (FP64)",
                      "runs": out}), flush=True)
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--maxiter", type=int, default=3000)
    ap.add_argument("--no-cpu", action="store_true", help="skip the CPU oracle baseline")
    ap.add_argument("--config", default="ci2m",
                    choices=["ci2m", "batched", "cfg1", "dense", "gram", "damping", "precond"],
                    help="ci2m: the headline workload; batched: the 256-problem serving workload; "
                         "cfg1 / dense: the n=4096 sparse and n=8192 dense configurations (side lines); "
                         "gram: the FP32 Gram kernels at n=2e6; damping: learned vs damped diagonal "
                         "preconditioners on held-out matrices; precond: diagonal, tridiagonal and learned "
                         "preconditioners as in the paper's Table 1 (side lines)")
    ap.add_argument("--nprob", type=int, default=256)
    ap.add_argument("--profile", action="store_true",
                    help="profiling run: time the mixed solves only (no FP64 comparison, e2e or CPU legs)")
    ap.add_argument("--n", type=int, default=N_ROWS, help="rows of the CI-like matrix (profiling runs only)")
    ap.add_argument("--threads", type=int, default=32)
    ap.add_argument("--fp64-runs", type=int, default=3, help="plain FP64 solves timed (median reported)")
    args = ap.parse_args()
    if args.n != N_ROWS and not args.profile:
        ap.error("--n changes the workload: only for --profile runs")
    if args.config == "batched":
        return run_batched(args)
    if args.config in ("cfg1", "dense"):
        return run_small_config(args)
    if args.config == "gram":
        return run_gram_config(args)
    if args.config == "damping":
        return run_damping_config(args)
    if args.config == "precond":
        return run_precond_config(args)
    if args.impl == "reference":
        return run_reference(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
