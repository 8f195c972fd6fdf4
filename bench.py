#!/usr/bin/env python
"""Benchmark: supernodal sparse Cholesky factor + solve on one GB300 (per rank).

Workload (the N=1 line): 3D 7-point variable-coefficient Laplacian on a 64^3
grid (n = 262,144), conductances log-uniform in [1e-2, 1e2], diagonal = incident
sum + 1e-6, geometric nested-dissection ordering; FP64 factor + solve with 8
right-hand sides U(-1, 1). One step = value scatter + numeric factorization +
8-RHS forward/backward solve + logdet, inputs resident in HBM (the factor panels,
1.65 GB, exceed the 129 MB L2, so no flush is needed between steps).

value = symbolic factor flops (sum_j c_j^2) / step time, summed over ranks
(independent replicas: the single factorization does not shard).

`--impl reference` times the CPU oracle (the plain FP64 left-looking column
Cholesky, numeric factor on every host core) on the same 3D 64^3 workload: one
whole factorization split over the timed steps, then the 8-RHS solve.
"""
import argparse
import json
import os
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "factor GFLOP/s + factor/solve ms at ≤1e-10 backward error, mixed vs FP64"
WORKLOAD = "3D 7-point var-coef Laplacian 64^3 (n=262144), FP64 factor + 8-RHS solve"
NRHS = 8
# FP64 peak derived from unit counts: 152 SMs x 2 FP64 FMA/clk/SM x 2 flop x 2.07 GHz
FP64_PEAK_GFLOPS = 152 * 2 * 2 * 2.07
# binary64 products run as 28 bf16 slice products on the tensor cores
# (csrc/split_gemm.cuh); cuBLAS bf16 under the power cap where it was measured
SLICE_PRODUCTS = 28
BF16_SUSTAINED_TFLOPS = 1700.0
# DRAM bytes (read + write) per launch of the SYRK class on this workload, from
# the ncu capture summarised in profiles/k_sg_syrk_fp64_3d64_traffic.md
SYRK_TRAFFIC_PER_LAUNCH = 8.246e9 / 36


def _env_int(k, d):
    try:
        return int(os.environ.get(k, d))
    except ValueError:
        return d


class ClockSampler:
    """nvidia-smi clock/throttle sampling during the timed region."""

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None
        self.lines = []

    def __enter__(self):
        q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), "--query-gpu=" + q,
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except Exception:
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
            except Exception:
                self.proc.kill()

    def summary(self):
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1])); mx = float(f[2])
            except ValueError:
                continue
            for nm, v in zip(names, f[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"]}
        return {"sm_mhz": float(np.median(sm)), "sm_max_mhz": mx, "reasons": sorted(reasons),
                "samples": len(sm)}


def bf16_sustained_tflops():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return float(json.load(f)["bf16_tflops_sustained"])
    except (OSError, KeyError, ValueError):
        return BF16_SUSTAINED_TFLOPS


def syrk_route(tc_products, achieved):
    """(on the tensor cores, kernels, peak, rate against it) of the SYRK class that ran
    at `achieved` binary64 GFLOP/s (or None), by the route that the handle reports."""
    if tc_products & 1:
        return (True, "k_sg_split_rows + k_sg_syrk", bf16_sustained_tflops() * 1e3,
                achieved * SLICE_PRODUCTS if achieved else None)
    return False, "k_syrk", FP64_PEAK_GFLOPS, achieved


def max_over_ranks(dist, values, device):
    """Element-wise maximum of per-rank timings (every rank gets the result)."""
    import torch
    if dist is None:
        return [float(v) for v in values]
    t = torch.tensor([float(v) for v in values], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return [float(v) for v in t.tolist()]


def replica_throughput(flops_per_replica, world, ms_max):
    """Whole-job GFLOP/s of `world` independent replicas, each doing one step of
    `flops_per_replica` flops, finishing within the slowest rank's `ms_max`."""
    return flops_per_replica * world / (ms_max * 1e-3) / 1e9


def _cpu_cores():
    try:
        return len(os.sched_getaffinity(0))
    except Exception:
        return os.cpu_count()


def oracle_sample(k=40, threads=1):
    """Oracle (as it stands) on the same generator at a bounded size: GFLOP/s.
    threads != 1 times its multi-threaded numeric factor (0 = all cores)."""
    import gridgen
    import oracle
    p = gridgen.laplacian_neumann_varcoef((k, k, k), 1e-2, 1e2, 1e-6, seed=2)
    b = gridgen.rhs_uniform(p.n, NRHS, seed=2)
    t = time.perf_counter()
    r = oracle.reference(p, b, threads=threads)
    dt = time.perf_counter() - t
    return r["sym"].flops() / dt / 1e9, dt, p.n


class OracleStepper:
    """The oracle on the benchmark workload itself (3D 64^3, 8 RHS): one
    multi-threaded numeric factorization split into `steps` pieces of
    elimination-tree heights with equal flops (the heights run in order, so the
    pieces together are exactly one factorization), the last piece followed by
    the 8-RHS solve and log det. Permutation and symbolic analysis are done
    before timing, as the GPU arm's analysis is."""

    def __init__(self, steps, threads, k=64):
        import gridgen
        import oracle
        self.oracle = oracle
        # k = 64 is the benchmark workload (gridgen.workload("3d64")); smaller k
        # only for quick checks of the harness
        self.p = gridgen.laplacian_neumann_varcoef((k, k, k), 1e-2, 1e2, 1e-6, seed=2)
        self.k = k
        self.b = gridgen.rhs_uniform(self.p.n, NRHS, seed=2)
        n = self.p.n
        self.B = oracle.permute(n, self.p["colptr"], self.p["rowind"], self.p["values"], self.p["perm"])
        self.sym = oracle.Symbolic(n, self.B[0], self.B[1])
        self.flops = float(self.sym.flops())
        self.threads = threads
        self.steps = max(int(steps), 1)
        self.S = None

    def start(self):
        bp, bi, bx = self.B
        self.S = self.oracle.StagedFactor(self.p.n, bp, bi, bx, threads=self.threads, sym=self.sym)
        w = np.cumsum(self.S.work())
        targets = w[-1] * np.arange(1, self.steps) / self.steps
        cuts = np.searchsorted(w, targets, side="left") + 1
        self.cuts = [0] + [int(c) for c in cuts] + [self.S.max_height + 1]
        self.piece = 0

    def step(self):
        """Run piece k; returns its wall seconds."""
        t = time.perf_counter()
        self.S.run(self.cuts[self.piece], self.cuts[self.piece + 1])
        self.piece += 1
        if self.piece == self.steps:
            fac = self.S.finish()
            self.x = fac.solve(self.p["perm"], self.b)
            self.logdet = fac.logdet()
            self.info = fac.info
        return time.perf_counter() - t


def run_reference(args, rank):
    if rank != 0:
        return
    cores = _cpu_cores()   # the oracle's multi-threaded numeric factor on every host core
    for _ in range(args.warmup):
        oracle_sample(16, threads=cores)
    st = OracleStepper(args.steps, cores, args.ref_grid)
    st.start()
    secs = [st.step() for _ in range(args.steps)]
    tot = float(np.sum(secs))
    value = st.flops / tot / 1e9
    eta = backward_error(st.p, st.b, st.x)
    sample = ("the whole benchmark workload: one oracle factorization of the 3D %d^3 matrix (numeric factor on "
              "%d threads) split over the %d timed steps by elimination-tree heights of equal flops, the last step "
              "also solving the 8 right-hand sides and taking log det; warm-up steps factor a 16^3 grid"
              % (args.ref_grid, cores, args.steps))
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": "GFLOP/s",
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * tot / args.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": WORKLOAD if args.ref_grid == 64 else "3D 7-point var-coef Laplacian %d^3 "
                       "(harness check, not the benchmark)" % args.ref_grid, "grid": args.ref_grid, "nrhs": NRHS,
                       "precision": "fp64", "l2": "inputs larger than L2"},
            "cpu_baseline": {"value": value, "unit": "GFLOP/s", "cores": cores, "kind": "oracle, multi-threaded",
                             "sample": sample},
            "e2e": {"value": value, "unit": "GFLOP/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
            "backward_error": float(eta), "logdet": st.logdet, "factor_info": int(st.info)}
    print(json.dumps(line), flush=True)


def backward_error(p, b, x):
    """eta = ||b - A x||_inf / (||A||_inf ||x||_inf + ||b||_inf) with scipy on the host."""
    import scipy.sparse as sp
    n = p["n"]
    Al = sp.csc_matrix((p["values"], p["rowind"], p["colptr"]), shape=(n, n))
    A = Al + sp.tril(Al, -1).T
    anorm = abs(A).sum(axis=1).max()
    r = b - A @ x
    return (np.abs(r).max(axis=0) / (anorm * np.abs(x).max(axis=0) + np.abs(b).max(axis=0))).max()


def _timed(torch, st, fn, reps):
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    out = None
    ms = []
    for _ in range(reps):
        torch.cuda.synchronize()
        e0.record(st)
        out = fn()
        e1.record(st)
        torch.cuda.synchronize()
        ms.append(e0.elapsed_time(e1))
    return float(np.median(ms)), out


def mixed_run(P, torch, dev, p, b, precision, merge, reps, static_pivot=0):
    """Factor with a mixed mode, refine all right-hand sides to eta <= 1e-10."""
    opt = P.chol_default_options()
    opt.precision = precision
    opt.merge_growth = merge
    opt.static_pivot = static_pivot
    S = P.SparseCholesky(p.n, p["colptr"], p["rowind"], p["perm"], opt)
    st = torch.cuda.current_stream()
    vals = torch.as_tensor(p["values"], device=dev)
    nrhs = b.shape[1]
    B = torch.as_tensor(np.ascontiguousarray(b.T), device=dev).t()
    X = torch.zeros_like(B)
    S.factor(vals)
    P.chol_solve_refine(S.h, B, X, nrhs, 1e-10, 200)
    fms, _ = _timed(torch, st, lambda: S.factor(vals), reps)
    rms, res = _timed(torch, st, lambda: P.chol_solve_refine(S.h, B, X, nrhs, 1e-10, 200), reps)
    rc, iters, berr = res
    eta = backward_error(p, b, X.cpu().numpy())
    info = P.chol_get_info(S.h)
    S.close()
    return {"precision": {1: "fp32", 2: "tf32", 3: "bf16"}[precision], "factor_ms": fms, "refine_ms": rms,
            "total_ms": fms + rms, "refine_rc": rc, "iterations": iters, "backward_error": float(eta),
            "fp64_fallback_blocks": info.fp64_fallbacks, "perturbed_pivots": info.perturbed_pivots}


def mixed_vs_fp64(args, P, gridgen, torch, dev, p, b, vals, flops, factor_ms, solve_ms):
    """Mixed precision + binary64 refinement to eta <= 1e-10 against the plain
    binary64 factor + solve, on the benchmark workload and on the 3D 48^3 x 3
    27-point elasticity workload (BF16/TF32 updates)."""
    out = {}
    best = None
    for prec in (1, 2):
        r = mixed_run(P, torch, dev, p, b, prec, args.merge, 3)
        out.setdefault("3d64", {})[r["precision"]] = r
        if r["refine_rc"] == 0 and (best is None or r["total_ms"] < best["total_ms"]):
            best = r
    out["3d64"]["fp64_ms"] = factor_ms + solve_ms
    if best:
        out["3d64"]["best"] = best["precision"]
        out["3d64"]["speedup"] = (factor_ms + solve_ms) / best["total_ms"]
        out["3d64"]["mixed_gflops"] = flops / (best["total_ms"] * 1e-3) / 1e9
    if not args.skip_elasticity:
        pe = gridgen.workload("elast48")
        be = gridgen.rhs_uniform(pe.n, 1, seed=3)
        opt = P.chol_default_options()
        opt.merge_growth = args.merge
        S = P.SparseCholesky(pe.n, pe["colptr"], pe["rowind"], pe["perm"], opt)
        st = torch.cuda.current_stream()
        ve = torch.as_tensor(pe["values"], device=dev)
        Be = torch.as_tensor(np.ascontiguousarray(be.T), device=dev).t()
        S.factor(ve)
        f64, _ = _timed(torch, st, lambda: S.factor(ve), 1)
        Xe = Be.clone()
        s64, _ = _timed(torch, st, lambda: S.solve_(Xe), 1)
        eflops = S.info.flops
        eta64 = backward_error(pe, be, Xe.cpu().numpy())
        S.close()
        e = {"workload": "3D 48^3 x 3-dof 27-point elasticity-like (n=331776), 1 RHS", "flops": eflops,
             "fp64": {"factor_ms": f64, "solve_ms": s64, "total_ms": f64 + s64, "backward_error": float(eta64),
                      "factor_gflops": eflops / (f64 * 1e-3) / 1e9}}
        bestm = None
        for prec in (2, 3):
            r = mixed_run(P, torch, dev, pe, be, prec, args.merge, 2)
            e[r["precision"]] = r
            if r["refine_rc"] == 0 and (bestm is None or r["total_ms"] < bestm["total_ms"]):
                bestm = r
        if bestm:
            e["best"] = bestm["precision"]
            e["speedup"] = (f64 + s64) / bestm["total_ms"]
            e["mixed_gflops"] = eflops / (bestm["total_ms"] * 1e-3) / 1e9
        out["elast48"] = e
    return out


def batch_run(args, P, gridgen, torch, dev, rank=0, world=1, dist=None):
    """2,000 independent 2D 5-point Laplacians (sides U{16..96}, log-uniform
    weights in [0.1, 10], Dirichlet ghosts), one RHS each: one block-diagonal
    analysis, autotuned launch configuration (persistent cooperative kernel in a
    CUDA graph when it wins); FP64 factor + solve, and binary32 factor +
    refinement to eta <= 1e-10. With several ranks each takes its share of the
    systems (balanced by the n^1.5 work model, paper_2409_14009_gb300.shard)
    and the per-system log dets are all-gathered after the timed region."""
    from paper_2409_14009_gb300.shard import gather_results, partition_systems
    t0 = time.perf_counter()
    probs_all = gridgen.batch_2d(count=args.batch_count)
    mine = partition_systems([p.n for p in probs_all], world)[rank]
    probs = [probs_all[i] for i in mine]
    bd = gridgen.block_diagonal(probs)
    gen_s = time.perf_counter() - t0
    offs = bd["meta"]["offsets"].astype(np.int32)
    b = gridgen.rhs_uniform(bd.n, 1, seed=4)
    st = torch.cuda.current_stream()
    vals = torch.as_tensor(bd["values"], device=dev)
    out = {"workload": "batch of %d 2D 5-point Laplacians, sides U{16..96}, n_total=%d, 1 RHS each"
                       % (len(probs_all), sum(p.n for p in probs_all)),
           "rank_share": {"systems": len(probs), "n": int(bd.n)}}
    tuned = {}
    for prec, name, mode in ((0, "fp64", 0), (0, "fp64_rlb", 1), (1, "fp32", 0)):
        base = P.chol_default_options()
        base.precision = prec
        base.update_mode = mode   # fp64_rlb: updates straight into the ancestors, no assembly pass
        # analysis choices (one-CTA thresholds, relaxed merging) searched on every
        # 10th system of this rank's share, then the whole share analyzed with them
        t0 = time.perf_counter()
        rc, opt, sample_ms, hit = P.chol_tune_batch(len(offs) - 1, offs, bd["colptr"], bd["rowind"], bd["perm"],
                                                    vals, base, 10, None, st)
        assert rc == 0, rc
        tune_s = time.perf_counter() - t0
        opt.persistent, opt.use_graph = 0, 0
        tuned[name] = {"small_max_cols": opt.small_max_cols, "small_max_panel": opt.small_max_panel,
                       "small_max_rows": opt.small_max_rows, "merge_growth": opt.merge_growth,
                       "search_s": tune_s, "sample_factor_ms": sample_ms}
        t0 = time.perf_counter()
        rc, h = P.chol_analyze_batch(len(offs) - 1, offs, bd["colptr"], bd["rowind"], bd["perm"], opt)
        ana_s = time.perf_counter() - t0
        assert rc == 0, rc
        info = P.chol_get_info(h)
        rc = P.chol_autotune(h, vals, st)
        assert rc == 0, rc
        info = P.chol_get_info(h)
        B = torch.as_tensor(np.ascontiguousarray(b.T), device=dev).t()
        X = torch.zeros_like(B)
        if dist:
            dist.barrier()
        fms, rcs = _timed(torch, st, lambda: P.chol_factor(h, vals, st), 5)
        assert rcs == 0, rcs
        if prec == 0:
            def solve():
                X.copy_(B)
                return P.chol_solve(h, X, 1, st)
            sms, _ = _timed(torch, st, solve, 5)
            iters = 0
        else:
            sms, res = _timed(torch, st, lambda: P.chol_solve_refine(h, B, X, 1, 1e-10, 50, st), 5)
            iters = res[1]
        fms, sms = max_over_ranks(dist, [fms, sms], dev)
        if dist:
            tfl = torch.tensor([info.flops], dtype=torch.float64, device=dev)
            dist.all_reduce(tfl)
            flops_all = float(tfl.item())
        else:
            flops_all = info.flops
        eta = backward_error(bd, b, X.cpu().numpy())
        # every rank learns every system's log det (the one exchange of the batch)
        rcl, lds = P.chol_logdet_batch(h, len(probs), st)
        ld_all, st_all = gather_results(dist, world, len(probs_all), mine, lds, [rcl] * len(probs), dev)
        out[name] = {"analyze_s": ana_s, "factor_ms": fms, "solve_ms": sms, "total_ms": fms + sms,
                     "refine_iterations": iters, "backward_error": float(eta),
                     "factor_gflops": flops_all / (fms * 1e-3) / 1e9,
                     "systems_per_s": len(probs_all) / ((fms + sms) * 1e-3),
                     "logdets_gathered": int(np.isfinite(ld_all).sum()), "ranks": world,
                     "autotuned": dict(tuned[name], persistent=bool(info.launch_mode & 1),
                                       graph=bool(info.launch_mode & 2),
                                       persistent_threads=info.persistent_threads,
                                       persistent_ctas_per_sm=info.persistent_ctas_per_sm),
                     "supernodes": info.nsuper_storage, "levels": info.nlevels}
        P.chol_destroy(h)
    out["flops"] = float(flops_all)
    out["generate_s"] = gen_s
    return out


def config1_run(args, P, gridgen, torch, dev):
    """The small 2D configuration: 5-point Dirichlet Laplacian on a 64^2 grid
    (n = 4,096, diagonal 4 + 1e-3), FP64 factor + one right-hand side U(-1, 1)
    + log det. About 2,000 supernodes, all at most 64 columns wide: the
    latency end of the method. Timed with direct launches and with the
    launch configuration the autotuner keeps (graph replay or the persistent
    cooperative kernel)."""
    p = gridgen.workload("2d64")
    b = gridgen.rhs_uniform(p.n, 1, seed=1)
    st = torch.cuda.current_stream()
    vals = torch.as_tensor(p["values"], device=dev)
    B = torch.as_tensor(b[:, 0].copy(), device=dev)
    X = torch.empty_like(B)
    out = {"workload": "2D 5-point Dirichlet Laplacian 64^2 (n=4096), FP64 factor + 1-RHS solve + log det"}
    for name, tune in (("direct", False), ("autotuned", True)):
        rc, h = P.chol_analyze(p.n, p["colptr"], p["rowind"], p["perm"])
        assert rc == 0, rc
        if tune:
            assert P.chol_autotune(h, vals, st) == 0
        info = P.chol_get_info(h)
        ld = [0.0]

        def step():
            assert P.chol_factor(h, vals, st) == 0
            X.copy_(B)
            assert P.chol_solve(h, X, 1, st) == 0
            ld[0] = P.chol_logdet(h, st)[1]
        for _ in range(5):
            step()
        P.chol_get_stats(h, reset=True)
        reps = 50
        ms, _ = _timed(torch, st, step, reps)
        stats = P.chol_get_stats(h, reset=True)
        fms, _ = _timed(torch, st, lambda: P.chol_factor(h, vals, st), 20)
        X.copy_(B)
        sms, _ = _timed(torch, st, lambda: P.chol_solve(h, X, 1, st), 20)
        X.copy_(B)
        P.chol_solve(h, X, 1, st)
        torch.cuda.synchronize()
        eta = backward_error(p, b, X.cpu().numpy().reshape(-1, 1))
        out[name] = {"ms_per_step": ms, "factor_ms": fms, "solve_ms": sms,
                     "factor_gflops": info.flops / (fms * 1e-3) / 1e9,
                     "launches_per_step": int(sum(v["launches"] for v in stats.values())) // reps,
                     "backward_error": float(eta), "logdet": ld[0],
                     "launch_mode": {"persistent": bool(info.launch_mode & 1), "graph": bool(info.launch_mode & 2)},
                     "supernodes": info.nsuper_storage, "levels": info.nlevels}
        P.chol_destroy(h)
    out["flops"] = float(info.flops)
    return out


def rlb_run(args, P, torch, dev, p, b, vals, flops, rl_factor_ms, rl_u_doubles):
    """The right-looking blocked update (no update workspace) on the bench
    workload: FP64 factor + 8-RHS solve, timed like the RL factor."""
    opt = P.chol_default_options()
    opt.merge_growth = args.merge
    opt.update_mode = P.CHOL_UPDATE_RLB
    S = P.SparseCholesky(p.n, p["colptr"], p["rowind"], p["perm"], opt)
    st = torch.cuda.current_stream()
    B = torch.as_tensor(np.ascontiguousarray(b.T), device=dev).t()
    X = torch.empty_like(B)
    S.factor(vals)
    fms, _ = _timed(torch, st, lambda: S.factor(vals), 3)
    X.copy_(B)
    S.solve_(X)
    torch.cuda.synchronize()
    eta = backward_error(p, b, X.cpu().numpy())
    out = {"factor_ms": fms, "factor_gflops": flops / (fms * 1e-3) / 1e9, "backward_error": float(eta),
           "rl_factor_ms": rl_factor_ms, "update_workspace_bytes_saved": int(rl_u_doubles * 8)}
    S.close()
    return out


def adjoint_run(args, P, gridgen, torch, dev):
    """Differentiable solve: 3D 48^3 7-point Dirichlet Laplacian (n=110,592),
    conductances log-uniform in [1e-2, 1e2], 16 RHS; loss = sum w^T x + log det A.
    Forward = factor + 16-RHS solve + logdet; backward = chol_adjoint (two
    triangular solves + selected inverse + per-nonzero gradient)."""
    p = gridgen.workload("3d48")
    b = gridgen.rhs_uniform(p.n, 16, seed=5)
    w = gridgen.rhs_normal(p.n, 16, seed=6)
    opt = P.chol_default_options()
    opt.merge_growth = args.merge
    S = P.SparseCholesky(p.n, p["colptr"], p["rowind"], p["perm"], opt)
    st = torch.cuda.current_stream()
    vals = torch.as_tensor(p["values"], device=dev)
    B = torch.as_tensor(np.ascontiguousarray(b.T), device=dev).t()
    W = torch.as_tensor(np.ascontiguousarray(w.T), device=dev).t()
    X = torch.empty_like(B)
    bbar = torch.empty_like(B)
    grad = torch.empty(len(p["rowind"]), dtype=torch.float64, device=dev)

    def forward():
        S.factor(vals)
        X.copy_(B)
        S.solve_(X)
        return S.logdet()

    def backward():
        return P.chol_adjoint(S.h, W, X, 16, 1.0, bbar, grad, st)

    forward(); backward()
    fms, _ = _timed(torch, st, forward, 3)
    bms, rc = _timed(torch, st, lambda: (forward(), backward())[1], 3)
    S.close()
    return {"workload": "3D 48^3 7-point Dirichlet Laplacian (n=110592), 16 RHS, loss = sum w^T x + log det A",
            "forward_ms": fms, "forward_plus_backward_ms": bms, "backward_ms": bms - fms, "rc": rc,
            "factor_flops": float(S.info.flops)}


def run_ours(args, rank, world, local_rank):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import gridgen
    import paper_2409_14009_gb300 as P
    torch.cuda.set_device(local_rank)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    dev = torch.device("cuda", local_rank)
    p = gridgen.workload(args.workload)
    b = gridgen.rhs_uniform(p.n, NRHS, seed=2)
    opt = P.chol_default_options()
    opt.merge_growth = args.merge
    t_ana = time.perf_counter()
    S = P.SparseCholesky(p.n, p["colptr"], p["rowind"], p["perm"], opt)
    analyze_ms = 1e3 * (time.perf_counter() - t_ana)   # host symbolic analysis, once per pattern
    flops = S.info.flops
    st = torch.cuda.current_stream()
    vals = torch.as_tensor(p["values"], device=dev)
    B = torch.as_tensor(np.ascontiguousarray(b.T), device=dev).t()   # column-major n x 8
    X = torch.empty_like(B)
    ld = [0.0]

    def step():
        S.factor(vals)
        X.copy_(B)
        S.solve_(X)
        ld[0] = S.logdet()

    for _ in range(max(args.warmup, 0)):
        step()
    torch.cuda.synchronize()
    # time the SYRK class (the most flops of a class, and alone on the GPU while it
    # runs) inside the timed region; per-launch events on one class only keep the
    # step's overhead small
    P.chol_profile(S.h, 1 << P.KERNEL_CLASSES.index("syrk"))
    P.chol_get_stats(S.h, reset=True)
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    with ClockSampler(local_rank) as clk:
        if dist:
            dist.barrier()
        torch.cuda.synchronize()
        e0.record(st)
        tf = []
        for _ in range(args.steps):
            step()
        e1.record(st)
        torch.cuda.synchronize()
        if dist:
            dist.barrier()
    ms = e0.elapsed_time(e1) / args.steps
    stats = P.chol_get_stats(S.h, reset=True)
    P.chol_profile(S.h, 0)
    launches = int(sum(v["launches"] for v in stats.values()))
    # factor-only and solve-only times (separate, untimed-for-value passes)
    f0 = torch.cuda.Event(enable_timing=True); f1 = torch.cuda.Event(enable_timing=True)
    f0.record(st); S.factor(vals); f1.record(st); torch.cuda.synchronize()
    factor_ms = f0.elapsed_time(f1)
    X.copy_(B)
    f0.record(st); S.solve_(X); f1.record(st); torch.cuda.synchronize()
    solve_ms = f0.elapsed_time(f1)
    eta = backward_error(p, b, X.cpu().numpy())
    # end to end through the C ABI with host buffers: chol_factor_solve_host
    # copies the values and right-hand sides in, factors, solves, takes log
    # det and copies X out, every step
    hv = torch.as_tensor(p["values"]).pin_memory()
    hb = torch.as_tensor(np.ascontiguousarray(b.T)).pin_memory()   # column-major n x 8
    hx = torch.empty_like(hb).pin_memory()

    def e2e_step():
        rc, ld_ = P.chol_factor_solve_host(S.h, hv, hb, hx, NRHS, True, st)
        assert rc == 0, rc
        return ld_
    e2e_step()
    torch.cuda.synchronize()
    f0.record(st)
    for _ in range(args.steps):
        ld_e2e = e2e_step()
    f1.record(st)
    torch.cuda.synchronize()
    e2e_ms = f0.elapsed_time(f1) / args.steps
    eta_e2e = backward_error(p, b, hx.numpy().T)
    mixed = None if args.no_mixed else mixed_vs_fp64(args, P, gridgen, torch, dev, p, b, vals, flops,
                                                         factor_ms, solve_ms)
    batch = None if args.no_batch else batch_run(args, P, gridgen, torch, dev, rank, world, dist)
    config1 = None if args.no_config1 else config1_run(args, P, gridgen, torch, dev)
    adjoint = None if args.no_adjoint else adjoint_run(args, P, gridgen, torch, dev)
    rlb = None if args.no_rlb else rlb_run(args, P, torch, dev, p, b, vals, flops, factor_ms,
                                           S.info.update_doubles)
    ms, e2e_ms = max_over_ranks(dist, [ms, e2e_ms], dev)
    if rank == 0:
        ds = stats["syrk"]
        achieved = ds["flops"] / (ds["ms"] * 1e-3) / 1e9 if ds["ms"] > 0 else None
        stored_ratio = S.info.flops_stored / flops
        rc_p, dfma, dfma_ghz = P.chol_probe_fp64(0, 3)
        rc_q, dmma, dmma_ghz = P.chol_probe_fp64(1, 3)
        tensor, kernel, peak, done = syrk_route(P.chol_get_info(S.h).tc_products, achieved)
        roof = {"bound": "tensor" if tensor else "alu", "kernel": kernel,
                # tensor: bf16 flops of the slice products, splitting included in the time
                "achieved": done, "peak": peak, "unit": "GFLOP/s",
                "frac": (done / peak) if done else None,
                "fp64_gflops": achieved, "fp64_pipe_peak": FP64_PEAK_GFLOPS,
                # the kernel's flops count the explicit zeros of relaxed merging;
                # the method's own share scales by the symbolic / stored ratio
                "frac_symbolic": (done / peak / stored_ratio) if done else None,
                "traffic": SYRK_TRAFFIC_PER_LAUNCH if tensor else None,
                "traffic_source": "profiles/k_sg_syrk_fp64_3d64_traffic.md (ncu dram__bytes_read/write.sum of the "
                                  "SYRK class of one 64^3 factorization, per launch)",
                "peak_source": "MEASURED_PEAKS.json bf16_tflops_sustained (cuBLAS bf16)" if tensor else
                               "derived: 152 SMs x 2 FP64 FMA/clk x 2.07 GHz (FP64 DFMA pipe); measured beside it "
                               "by chol_probe_fp64 (profiles/fp64_peak_probe.md)",
                "peak_measured": {"dfma": dfma if rc_p == 0 else None, "dfma_sm_ghz": dfma_ghz,
                                  "dmma": dmma if rc_q == 0 else None, "dmma_sm_ghz": dmma_ghz,
                                  "dfma_at_2070mhz": (dfma * 2.07 / dfma_ghz) if (rc_p == 0 and dfma_ghz > 0)
                                  else None},
                "launches": ds["launches"], "ms_total": ds["ms"]}
        cpu = cpu_mt = None
        if world == 1 and not args.no_cpu_baseline:
            v, dt, n = oracle_sample(args.cpu_grid)
            cpu = {"value": v, "unit": "GFLOP/s", "cores": 1, "kind": "oracle",
                   "sample": "oracle FP64 factor+solve(8 RHS), same generator on a %d^3 grid (n=%d), %.1f s"
                             % (args.cpu_grid, n, dt)}
            # the same loops on every host core, on the benchmark workload itself
            cores = _cpu_cores()
            ost = OracleStepper(1, cores)
            ost.start()
            dtt = ost.step()
            cpu_mt = {"value": ost.flops / dtt / 1e9, "unit": "GFLOP/s", "cores": cores,
                      "kind": "oracle, multi-threaded", "same_config": True,
                      "sample": "the whole 3D 64^3 workload: numeric factor on %d threads + 8-RHS solve + log det, "
                                "%.1f s (permutation and symbolic analysis not timed)" % (cores, dtt),
                      "backward_error": float(backward_error(ost.p, ost.b, ost.x))}
        line = {"metric": METRIC, "value": replica_throughput(flops, world, ms), "unit": "GFLOP/s",
                "n_gpus": world, "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms,
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
                "data": "synthetic",
                "config": {"workload": WORKLOAD if args.workload == "3d64" else args.workload,
                           "nrhs": NRHS, "precision": "fp64",
                           "merge_growth": args.merge, "supernodes": S.info.nsuper_storage,
                           "flops_stored_over_symbolic": S.info.flops_stored / flops,
                           "parallelism": "replicas" if world > 1 else "single",
                           "l2": "inputs larger than L2 (panels 1.65 GB)"},
                "analyze_ms": analyze_ms, "factor_ms": factor_ms, "solve_ms": solve_ms,
                "factor_gflops": flops / (factor_ms * 1e-3) / 1e9, "flops": flops,
                "backward_error": float(eta), "logdet": ld[0],
                "e2e": {"value": replica_throughput(flops, world, e2e_ms), "unit": "GFLOP/s",
                        "ms_per_step": e2e_ms, "h2d_bytes_per_step": int(hv.numel() * 8 + hb.numel() * 8),
                        "d2h_bytes_per_step": int(hx.numel() * 8 + 8 + 4),
                        "api": "chol_factor_solve_host (pinned host values and right-hand sides in, X and "
                               "log det out; factor + 8-RHS solve + log det per step)",
                        "backward_error": float(eta_e2e), "logdet": ld_e2e},
                "gpu_launches": launches // max(args.steps, 1) * args.steps,
                "roofline": roof, "cpu_baseline": cpu, "cpu_baseline_threads": cpu_mt, "clocks": clk.summary(),
                "mixed_vs_fp64": mixed, "batch": batch, "adjoint": adjoint, "rlb": rlb, "config1_2d64": config1}
        print(json.dumps(line), flush=True)
    S.close()
    if dist:
        dist.destroy_process_group()


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--cpu-grid", type=int, default=40)
    ap.add_argument("--ref-grid", type=int, default=64,
                    help="grid side of the reference arm (64 = the benchmark workload itself)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-mixed", action="store_true", help="skip the mixed-precision comparison")
    ap.add_argument("--skip-elasticity", action="store_true")
    ap.add_argument("--no-batch", action="store_true", help="skip the 2,000-system batch")
    ap.add_argument("--batch-count", type=int, default=2000)
    ap.add_argument("--no-adjoint", action="store_true", help="skip the differentiable-solve workload")
    ap.add_argument("--no-rlb", action="store_true", help="skip the right-looking blocked (RLB) factor")
    ap.add_argument("--no-config1", action="store_true", help="skip the 2D 64^2 configuration")
    ap.add_argument("--workload", default="3d64", choices=["3d64", "3d48"],
                    help="3d64 is the benchmark; 3d48 is the smaller case used for ncu captures")
    ap.add_argument("--merge", type=float, default=0.1,
                    help="relaxed supernode merging budget (fraction of nnz(L))")
    args = ap.parse_args()
    rank = _env_int("RANK", 0)
    world = _env_int("WORLD_SIZE", 1)
    local_rank = _env_int("LOCAL_RANK", 0)
    if args.impl == "reference":
        run_reference(args, rank)
        return
    run_ours(args, rank, world, local_rank)


if __name__ == "__main__":
    main()
