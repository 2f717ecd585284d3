#!/usr/bin/env python
"""Benchmark: PCG solve of the GDML force-kernel system (K + lambda I) alpha = y on GB300.

One step = the whole hot path on one synthetic system: kernel setup
(descriptors, Jacobians, distance tables, diag K), preconditioner build
(inducing-column selection + Nystrom / incomplete-Cholesky factor + Woodbury
core) and the PCG solve to TRUE relative residual 1e-8 (Sec. 2.1, Eqs. 1-5,
Alg. 1).  Default workload: N=42 atoms, M=5000 geometries (n = 630,000,
D = 861), ridge-leverage-score preconditioner with k = 5000, length scale 30,
lambda 1e-9, in the OZAKI form (FP64-class contractions on the BF16 tensor cores).

Prints ONE JSON line (rank 0): the headline seconds per solve with inputs resident in
HBM, the same through host buffers (e2e), the matvec and Woodbury-apply rooflines, the
matvec of every form at this size and every form solved to the end on the 63,000-unknown
system, and the FP64 CPU oracle's extrapolated time on this host.  --impl reference
times that oracle alone (bounded samples, extrapolated to the full solve).
Multi-GPU (torchrun): replicas only -- every rank solves its own copy of the
system; no data-path collective exists for a single system here.
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
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "PCG seconds to rel. residual 1e-8 and matvec TFLOP/s, mixed vs FP64, 1 GB300"
RTOL = 1e-8


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=1)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="gdml", choices=["gdml", "reference"])
    ap.add_argument("--workload", default="mol42_m5000")
    ap.add_argument("--forms-workload", default="aspirin21_m1000",
                    help="system on which every form is solved to the end (FP64 takes minutes at n = 630,000)")
    ap.add_argument("--precision", default="ozaki", choices=["fp64", "tf32", "bf16", "df64", "ozaki"],
                    help="headline form (df64: double-float contractions on the FP32 lanes; ozaki: exact "
                         "BF16 residues on the tensor cores; both FP64-class, FP64 true-residual restarts)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-forms", action="store_true", help="skip the per-precision comparison solves")
    ap.add_argument("--only", default="solve", choices=["solve", "matvec", "apply", "passes", "build"],
                    help="time one operation alone (small runs for profiling); passes: the two staged "
                         "passes of the DF64/OZAKI apply on a random FP32 factor of the workload's n x k")
    ap.add_argument("--rows", type=int, default=1, choices=[1, 128, 256],
                    help="--only passes: row-chunk size of the staged passes (1: automatic)")
    ap.add_argument("--suite", default=None, choices=["batched", "learned", "sym"],
                    help="many uneven systems: per-system solves vs one batched graph solve")
    ap.add_argument("--suite-count", type=int, default=64)
    ap.add_argument("--suite-mmax", type=int, default=2000, help="cap on M (geometries) per system")
    ap.add_argument("--suite-maxiter", type=int, default=2000, help="PCG iteration cap per system in the suite")
    ap.add_argument("--cpu-sample", default=None, help=argparse.SUPPRESS)  # internal: 1-core oracle sample
    ap.add_argument("--ref-iters", type=int, default=0,
                    help="PCG iterations the oracle's sampled cost is extrapolated with (default: REF_ITERS)")
    return ap.parse_args()


# tensor-core products per FP64-equivalent product: the OZAKI form multiplies residues
# modulo 14 numbers for each one
TC_PRODUCTS = {"fp64": 1, "df64": 1, "tf32": 1, "bf16": 1, "ozaki": 14}


# ----------------------------------------------------------------- helpers
class ClockSampler:
    """nvidia-smi clocks / throttle reasons sampled every 200 ms while running."""

    FIELDS = ["index", "clocks.sm", "clocks.max.sm", "power.draw", "clocks_event_reasons.active",
              "clocks_event_reasons.hw_slowdown", "clocks_event_reasons.hw_thermal_slowdown",
              "clocks_event_reasons.sw_thermal_slowdown", "clocks_event_reasons.sw_power_cap"]

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.rows = []
        self.proc = None

    def __enter__(self):
        if self.gpu < 0:  # not sampled
            return self
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={','.join(self.FIELDS)}", "--format=csv,noheader,nounits", "-lms",
                 "200", "-i", str(self.gpu)], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except OSError:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            parts = [p.strip() for p in line.split(",")]
            if len(parts) == len(self.FIELDS):
                self.rows.append(parts)

    def __exit__(self, *exc):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        if not self.rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unavailable"]}
        sm = [float(r[1]) for r in self.rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in self.rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in self.rows for i in range(4) if r[5 + i].lower() == "active"})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(self.rows)}


def measured_peaks():
    try:
        return json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
    except (OSError, ValueError):
        return {}


# ------------------------------------------------------------- GPU arm
def run_op(args):
    """--only matvec|apply: W untimed + K timed calls of one operation, one JSON line."""
    import torch

    from paper_2212_12737_gb300 import gdml, synth

    torch.cuda.set_device(0)
    dev = torch.device("cuda", 0)
    w = synth.workload(args.workload)
    if args.only == "passes":  # the library's test hook on a random factor (its columns contiguous)
        g = torch.Generator(device=dev).manual_seed(0)
        Lc = torch.randn(w.k, w.n, device=dev, generator=g).float()
        r = torch.randn(w.n, dtype=torch.float64, device=dev, generator=g)
        u = torch.randn(w.k, dtype=torch.float64, device=dev, generator=g)
        fn = lambda: gdml.test_df_passes(Lc.t(), r, u, w.lam, staged=args.rows)
        for _ in range(args.warmup):
            fn()
        torch.cuda.synchronize(dev)
        t0 = time.perf_counter()
        for _ in range(args.steps):
            fn()
        torch.cuda.synchronize(dev)
        ms = (time.perf_counter() - t0) * 1e3 / args.steps
        print(json.dumps({"op": "passes", "workload": args.workload, "rows": args.rows, "n": w.n, "k": w.k,
                          "host_ms_per_call": ms, "note": "includes the hook's scratch allocation; use ncu "
                          "kernel durations"}), flush=True)
        return
    ctx = gdml.kernel_setup(torch.from_numpy(w.R).to(dev), w.sigma, w.lam, precision=args.precision)
    if args.only == "build":  # preconditioner builds (Algorithm 1 / Nystrom + Woodbury core), host-timed
        ts = []
        for it in range(args.warmup + args.steps):
            torch.cuda.synchronize(dev)
            t0 = time.perf_counter()
            ctx.precond_build(w.select, w.k, seed=2)
            torch.cuda.synchronize(dev)
            if it >= args.warmup:
                ts.append(time.perf_counter() - t0)
        print(json.dumps({"op": "build", "workload": args.workload, "precision": args.precision,
                          "select": w.select, "k": w.k, "s": min(ts) if ts else None}), flush=True)
        ctx.destroy()
        return
    v = torch.randn(w.n, dtype=torch.float64, device=dev)
    out = torch.empty_like(v)
    if args.only == "apply":
        ctx.precond_build(w.select, w.k, seed=2)
        fn = lambda: ctx.precond_apply(v, out)
    else:
        fn = lambda: ctx.matvec(v, out)
    for _ in range(args.warmup):
        fn()
    st = torch.cuda.current_stream(dev)
    s = torch.cuda.Event(enable_timing=True)
    e = torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize(dev)
    s.record(st)
    for _ in range(args.steps):
        fn()
    e.record(st)
    torch.cuda.synchronize(dev)
    ms = s.elapsed_time(e) / args.steps
    D = w.N * (w.N - 1) // 2
    print(json.dumps({"op": args.only, "workload": args.workload, "precision": args.precision, "ms": ms,
                      "matvec_tflops": 6.0 * w.M * w.M * D / ms / 1e9 if args.only == "matvec" else None,
                      "apply_gbs": (2.0 * w.n * w.k * (4 if args.precision in ("df64", "ozaki") else 8)
                                    + 3.0 * w.k * w.k * 8) / ms / 1e6 if args.only == "apply" else None}),
          flush=True)
    ctx.destroy()


def run_suite(args):
    """Many uneven systems (N in {9,12,15,21,42}, M in [100, mmax], sigma in
    {5,10,20,40}, lambda in {1e-10,1e-8}, uniform k = M/10): per-system FP64 solves
    one after another (the reference launches) against the mixed-precision OZAKI form,
    per system and as one batched graph solve, each context autotuned first (the FP64
    batched solve is the same graph machinery and is not repeated here)."""
    import torch

    from paper_2212_12737_gb300 import gdml, synth

    torch.cuda.set_device(0)
    dev = torch.device("cuda", 0)
    suite = synth.batched_suite(args.suite_count, mmax=args.suite_mmax)
    cache = os.path.join(ROOT, "paper_2212_12737_gb300", "lib", "tuning.json")
    ys = [torch.from_numpy(w.y).to(dev) for w in suite]
    res = {"suite": "batched", "systems": len(suite), "total_unknowns": sum(w.n for w in suite),
           "mmax": args.suite_mmax, "max_iter": args.suite_maxiter}
    for prec in ("fp64", "ozaki"):
        ctxs = []
        t0 = time.perf_counter()
        for w in suite:
            c = gdml.kernel_setup(torch.from_numpy(w.R).to(dev), w.sigma, w.lam, precision=prec)
            c.autotune(cache)
            c.precond_build("uniform", w.k, seed=2)
            ctxs.append(c)
        torch.cuda.synchronize(dev)
        t_setup = time.perf_counter() - t0
        t0 = time.perf_counter()
        seq = []
        for c, y in zip(ctxs, ys):
            _, it, rel, _ = c.pcg_solve(y, rtol=RTOL, max_iter=args.suite_maxiter, raise_on_nonconvergence=False)
            seq.append((it, rel))
        torch.cuda.synchronize(dev)
        t_seq = time.perf_counter() - t0
        res[prec] = {"setup_autotune_build_s": t_setup, "per_system_solves_s": t_seq,
                     "iters_total": int(sum(it for it, _ in seq)),
                     "converged": int(sum(rel <= RTOL for _, rel in seq)), "max_relres": max(rel for _, rel in seq)}
        if prec == "ozaki":  # the mixed form also as one batched graph solve
            t0 = time.perf_counter()
            _, its, rels = gdml.pcg_solve_batched(ctxs, ys, rtol=RTOL, max_iter=args.suite_maxiter,
                                                  raise_on_nonconvergence=False)
            torch.cuda.synchronize(dev)
            res[prec].update({"batched_graph_solve_s": time.perf_counter() - t0, "batched_iters_total": int(sum(its)),
                              "batched_converged": int(sum(r <= RTOL for r in rels)),
                              "batched_same_iterations_as_per_system": all(a == b[0] for a, b in zip(its, seq))})
        for c in ctxs:
            c.destroy()
    res["mixed_batched_vs_fp64_per_system_speedup"] = (res["fp64"]["per_system_solves_s"]
                                                        / res["ozaki"]["batched_graph_solve_s"])
    print(json.dumps(res), flush=True)


def run_learned(args):
    """Learned inducing-column scorer: train on EXACT per-geometry ridge-leverage
    labels of training systems of the same molecule (other noise seeds) at reduced M
    (M = 100: exact scores need a dense eigendecomposition of K), select k columns for
    the headline system, and compare PCG iterations / solve time with pivoted Cholesky
    (the fallback and referee)."""
    import torch

    from paper_2212_12737_gb300 import gdml, synth

    torch.cuda.set_device(0)
    dev = torch.device("cuda", 0)
    base = dict(synth.WORKLOADS[args.workload])
    k = base["k"]
    t0 = time.perf_counter()
    Xs, ys = [], []
    m_train = 100
    n_train = min(args.suite_count, 20)
    for s in range(n_train):
        cfg = dict(base)
        w = synth.make_workload(f"train{s}", cfg["N"], m_train, cfg["noise"], cfg["sigma"], cfg["lam"],
                                min(k, 3 * cfg["N"] * m_train), "uniform", template_seed=0, noise_seed=100 + s)
        c = gdml.kernel_setup(torch.from_numpy(w.R).to(dev), w.sigma, w.lam)
        Xs.append(c.descriptors())
        ys.append(gdml.geometry_labels(c, exact=True))
        c.destroy()
    torch.cuda.synchronize(dev)
    t_labels = time.perf_counter() - t0
    X = torch.cat(Xs)
    y = torch.cat(ys)
    sc = gdml.Scorer(X.shape[1], 256, seed=0)
    sc.fit_scaling(X, y)
    t0 = time.perf_counter()
    loss = sc.train(X, y, epochs=30, batch=256, lr=1e-3)
    torch.cuda.synchronize(dev)
    t_train = time.perf_counter() - t0
    w = synth.workload(args.workload)
    R = torch.from_numpy(w.R).to(dev)
    yv = torch.from_numpy(w.y).to(dev)

    def timed(fn):
        torch.cuda.synchronize(dev)
        t = time.perf_counter()
        out = fn()
        torch.cuda.synchronize(dev)
        return time.perf_counter() - t, out

    prec = args.precision  # the headline form (OZAKI by default)

    def pivchol():
        c = gdml.kernel_setup(R, w.sigma, w.lam, precision=prec)
        c.precond_build("pivchol", k)
        _, it, rel, _ = c.pcg_solve(yv, rtol=RTOL, max_iter=20000, raise_on_nonconvergence=False)
        c.destroy()
        return it, rel

    def learned(referee):
        c = gdml.kernel_setup(R, w.sigma, w.lam, precision=prec)
        _, it, rel, used = gdml.solve_learned(c, sc, yv, k, referee_iters=referee)
        c.destroy()
        return it, rel, used

    t_pc, (it_pc, rel_pc) = timed(pivchol)
    t_l, (it_l, rel_l, used) = timed(lambda: learned(it_pc))
    # learned without the referee's cap, to report its own iteration count
    c = gdml.kernel_setup(R, w.sigma, w.lam, precision=prec)
    c.precond_build_scored(sc.predict(c.descriptors()), k)
    _, it_raw, rel_raw, _ = c.pcg_solve(yv, rtol=RTOL, max_iter=20000, raise_on_nonconvergence=False)
    c.destroy()
    c = gdml.kernel_setup(R, w.sigma, w.lam, precision=prec)
    c.precond_build("uniform", k, seed=2)
    _, it_u, rel_u, _ = c.pcg_solve(yv, rtol=RTOL, max_iter=20000, raise_on_nonconvergence=False)
    c.destroy()
    print(json.dumps({"suite": "learned", "workload": args.workload, "precision": prec, "k": k,
                      "train_systems": n_train,
                      "train_geometries_per_system": m_train, "labels": "exact ridge leverage scores",
                      "label_s": t_labels, "train_s": t_train, "train_loss": loss,
                      "pivchol": {"s": t_pc, "iters": it_pc, "relres": rel_pc},
                      "learned": {"s": t_l, "iters": it_l, "relres": rel_l, "used": used,
                                  "iters_without_referee": it_raw, "relres_without_referee": rel_raw},
                      "uniform": {"iters": it_u, "relres": rel_u}}), flush=True)
    sc.destroy()


def run_sym(args):
    """sGDML: the symmetric force kernel with the group S3 of atoms 0, 1, 2 (6 permutations, the
    size of a methyl group's symmetries) against the plain kernel on the same system: matvec time
    in FP64 and OZAKI, and the OZAKI solve (setup, pivoted-Cholesky build, PCG to 1e-8)."""
    import itertools

    import torch

    from paper_2212_12737_gb300 import gdml, synth

    torch.cuda.set_device(0)
    dev = torch.device("cuda", 0)
    w = synth.workload(args.workload)
    idn = list(range(w.N))
    group = []
    for p3 in itertools.permutations((0, 1, 2)):
        g = list(idn)
        g[0], g[1], g[2] = p3
        group.append(g)
    R = torch.from_numpy(w.R).to(dev)
    y = torch.from_numpy(w.y).to(dev)
    v = torch.randn(w.n, dtype=torch.float64, device=dev)
    out = torch.empty_like(v)
    st = torch.cuda.current_stream(dev)

    def mv_ms(ctx, reps):
        for _ in range(2):
            ctx.matvec(v, out)
        s = torch.cuda.Event(enable_timing=True)
        e = torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize(dev)
        s.record(st)
        for _ in range(reps):
            ctx.matvec(v, out)
        e.record(st)
        torch.cuda.synchronize(dev)
        return s.elapsed_time(e) / reps

    res = {"suite": "sym", "workload": f"{w.name}: n={w.n}, {w.select} k={w.k}, lambda={w.lam}", "S": len(group),
           "group": "S3 on atoms 0, 1, 2"}
    for prec in ("fp64", "ozaki"):
        for label, perms in (("plain", None), ("sym", group)):
            ctx = gdml.kernel_setup(R, w.sigma, w.lam, precision=prec, perms=perms)
            res[f"{prec}_{label}_matvec_ms"] = mv_ms(ctx, 3 if prec == "fp64" else 20)
            ctx.destroy()
    for label, perms in (("plain", None), ("sym", group)):
        torch.cuda.synchronize(dev)
        t0 = time.perf_counter()
        ctx = gdml.kernel_setup(R, w.sigma, w.lam, precision="ozaki", perms=perms)
        ctx.precond_build(w.select, w.k, seed=2)
        torch.cuda.synchronize(dev)
        t1 = time.perf_counter()
        _, it, rel, _ = ctx.pcg_solve(y, rtol=RTOL, max_iter=20000, raise_on_nonconvergence=False)
        t2 = time.perf_counter()
        ctx.tc_check()
        ctx.destroy()
        res[f"ozaki_{label}_solve"] = {"s": t2 - t0, "setup_build_s": t1 - t0, "pcg_s": t2 - t1, "iters": it,
                                       "relres": rel, "converged": rel <= RTOL}
    print(json.dumps(res), flush=True)


def max_over_ranks(t: float, world: int, device) -> float:
    """The job takes as long as its slowest rank: all-reduce MAX of t over the process group."""
    if world == 1:
        return t
    import torch
    import torch.distributed as dist
    tt = torch.tensor([t], dtype=torch.float64, device=device)
    dist.all_reduce(tt, op=dist.ReduceOp.MAX)
    return float(tt.item())


# DRAM bytes (dram__bytes_read.sum + dram__bytes_write.sum) per launch of the roofline's unit,
# from one ncu capture each (profiles/), keyed by (workload, precision, unit).  A unit whose
# kernels changed since the capture has no entry (traffic null).
NCU_TRAFFIC = {
    # profiles/woodbury_apply_dram_aspirin21_m1000_k2000_ozaki.md (cold-cache capture of one apply)
    ("aspirin21_m1000", "ozaki", "apply"): 1.1116e9,
    # the same capture scaled to n = 630,000, k = 5000: passes by n k, k x k core by k^2
    ("mol42_m5000", "ozaki", "apply"): 2.587e10,
}


def run_gpu(args):
    import numpy as np
    import torch
    import torch.distributed as dist

    from paper_2212_12737_gb300 import gdml, synth

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        dist.init_process_group("nccl")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    w = synth.workload(args.workload)
    M, N, n, k = w.M, w.N, w.n, w.k
    D = N * (N - 1) // 2
    R_h = torch.from_numpy(w.R).pin_memory()
    y_h = torch.from_numpy(w.y).pin_memory()
    R_d = R_h.to(dev)
    y_d = y_h.to(dev)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)  # > 129 MB L2
    stream = torch.cuda.current_stream(dev)

    def barrier():
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize(dev)

    def step(prec, R, y, wl=w, out_h=None, inner_levels=7):
        """one pass of the hot path: setup, preconditioner build, PCG to rtol (phases host-timed;
        every library call below already synchronises its stream before returning)"""
        t0 = time.perf_counter()
        ctx = gdml.kernel_setup(R, wl.sigma, wl.lam, precision=prec)
        torch.cuda.synchronize(dev)
        t1 = time.perf_counter()
        ctx.precond_build(wl.select, wl.k, seed=2)
        if inner_levels != 7:
            ctx.set_inner_levels(inner_levels)
        t2 = time.perf_counter()
        alpha, iters, rel, outer = ctx.pcg_solve(y, rtol=RTOL, max_iter=20000, raise_on_nonconvergence=False)
        t3 = time.perf_counter()
        if out_h is not None:
            out_h.copy_(alpha, non_blocking=True)
        ctx.destroy()
        return {"iters": iters, "relres": rel, "outer": outer, "setup_s": t1 - t0, "build_s": t2 - t1,
                "solve_s": t3 - t2}

    def timed(fn, steps, warmup, sample_clocks=True):
        info = None
        for _ in range(warmup):
            flush.fill_(1.0)
            info = fn()
        ts, infos = [], []
        barrier()
        with ClockSampler(local if sample_clocks else -1) as clk:
            for _ in range(steps):
                flush.fill_(2.0)  # untimed L2 flush between steps
                s = torch.cuda.Event(enable_timing=True)
                e = torch.cuda.Event(enable_timing=True)
                s.record(stream)
                info = fn()
                e.record(stream)
                torch.cuda.synchronize(dev)
                ts.append(s.elapsed_time(e) / 1e3)
                infos.append(info)
        barrier()
        t = max_over_ranks(sum(ts) / len(ts), world, dev)
        return t, infos, clk.summary()

    # headline: device-resident inputs
    n0 = gdml.launch_count()
    t_dev, infos, clocks = timed(lambda: step(args.precision, R_d, y_d), args.steps, args.warmup)
    launches = (gdml.launch_count() - n0) // (args.steps + args.warmup)
    head = infos[-1]

    # e2e: host inputs, H2D + D2H inside the timed region (the headline's warm-up already ran)
    alpha_h = torch.empty(n, dtype=torch.float64).pin_memory()

    def e2e_step():
        R = R_h.to(dev, non_blocking=True)
        y = y_h.to(dev, non_blocking=True)
        return step(args.precision, R, y, out_h=alpha_h)

    t_e2e, _, _ = timed(e2e_step, max(1, args.steps), 0, sample_clocks=False)

    def op_rate(ctx, fn, reps=20):
        for _ in range(3):
            fn()
        s = torch.cuda.Event(enable_timing=True)
        e = torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize(dev)
        s.record(stream)
        for _ in range(reps):
            fn()
        e.record(stream)
        torch.cuda.synchronize(dev)
        return s.elapsed_time(e) / 1e3 / reps

    v = torch.randn(n, dtype=torch.float64, device=dev)
    out = torch.empty_like(v)
    # the two per-iteration operations on one built context of the headline form
    ctx = gdml.kernel_setup(R_d, w.sigma, w.lam, precision=args.precision)
    mv_sec = op_rate(ctx, lambda: ctx.matvec(v, out))
    ctx.precond_build(w.select, k, seed=2)
    ap_sec = op_rate(ctx, lambda: ctx.precond_apply(v, out))
    ctx.destroy()

    def torch_peak(dtype, tf32=False, size=4096):
        torch.backends.cuda.matmul.allow_tf32 = tf32
        a = torch.randn(size, size, device=dev, dtype=dtype)
        b = torch.randn(size, size, device=dev, dtype=dtype)
        for _ in range(2):
            a @ b
        torch.cuda.synchronize(dev)
        best = 1e9
        for _ in range(3):
            s = torch.cuda.Event(enable_timing=True)
            e = torch.cuda.Event(enable_timing=True)
            s.record(stream)
            a @ b
            e.record(stream)
            torch.cuda.synchronize(dev)
            best = min(best, s.elapsed_time(e) / 1e3)
        torch.backends.cuda.matmul.allow_tf32 = False
        return 2.0 * size ** 3 / best / 1e12

    peaks = measured_peaks()
    if args.precision == "fp64":
        peak, peak_src, bound = torch_peak(torch.float64), "of measured (torch FP64 matmul 4096^3, this run)", "alu"
    elif args.precision == "df64":
        # double-float on the FP32 lanes: one multiply-add (2 flop) costs ~15 FP32
        # instructions where an FP32 FMA (also 2 flop) costs one, so the ceiling is
        # the measured FP32 SIMT matmul rate / 15
        peak = torch_peak(torch.float32, tf32=False, size=8192) / 15.0
        peak_src, bound = "of derived (torch FP32 SIMT matmul 8192^3 this run / 15 FP32 ops per double-float FMA)", "alu"
    elif args.precision == "tf32":
        peak, peak_src, bound = torch_peak(torch.float32, tf32=True, size=8192), \
            "of measured (torch TF32 matmul 8192^3, this run)", "tensor"
    else:  # ozaki (14 BF16 residue products per contraction on tcgen05) and bf16
        peak = peaks.get("bf16_tflops", 1900.0)
        peak_src, bound = ("of measured (MEASURED_PEAKS.json bf16_tflops, burst: the matvec is timed alone)"
                           if peaks else "of fallback"), "tensor"

    mv_flop = 6.0 * M * M * D * TC_PRODUCTS[args.precision]
    roof_matvec = {"kernel": f"force-kernel matvec, {args.precision}: one launch unit = projection + "
                             f"{'residue ' if args.precision == 'ozaki' else ''}contractions + beta + back-projection",
                   "bound": bound, "achieved": mv_flop / mv_sec / 1e12, "peak": peak, "unit": "TFLOP/s",
                   "frac": mv_flop / mv_sec / 1e12 / peak, "peak_source": peak_src,
                   "traffic": NCU_TRAFFIC.get((args.workload, args.precision, "matvec")),
                   "algorithmic_flop_per_launch": mv_flop,
                   "algorithmic_flop_note": ("14 BF16 residue products x 6 M^2 D" if args.precision == "ozaki"
                                             else "6 M^2 D"),
                   "fp64_equivalent_tflops": 6.0 * M * M * D / mv_sec / 1e12, "ms": mv_sec * 1e3}
    hbm = peaks.get("hbm_gbs", 6800.0)
    lbytes = 4 if args.precision in ("df64", "ozaki") else 8  # FP32-stored L_k in the double-float forms
    ap_bytes = 2.0 * n * k * lbytes  # the method's bytes: L_k read twice (L_k^T r and L_k u)
    core_bytes = 3.0 * k * k * 8    # the k x k core products (C^-1, C, C^-1), served from L2
    roof_apply = {"kernel": f"Woodbury apply (Eq. 4), {args.precision}: L_k^T r and L_k u passes + k x k core",
                  "bound": "hbm", "achieved": ap_bytes / ap_sec / 1e9, "peak": hbm, "unit": "GB/s",
                  "frac": ap_bytes / ap_sec / 1e9 / hbm,
                  "peak_source": "of measured (MEASURED_PEAKS.json hbm_gbs)" if peaks else "of fallback",
                  "traffic": NCU_TRAFFIC.get((args.workload, args.precision, "apply")),
                  "algorithmic_bytes_per_launch": ap_bytes,
                  "algorithmic_bytes_note": f"2 n k x {lbytes} B (L_k streamed twice); the k x k core "
                                            f"({core_bytes / 1e6:.0f} MB) is not counted",
                  "ms": ap_sec * 1e3}

    forms = {}
    forms_solve = {}
    if not args.no_forms and rank == 0:
        # matvec of every form at this workload (the metric's "matvec TFLOP/s, mixed vs FP64")
        for prec in ("fp64", "df64", "ozaki", "tf32", "bf16"):
            c2 = gdml.kernel_setup(R_d, w.sigma, w.lam, precision=prec)
            sec = op_rate(c2, lambda: c2.matvec(v, out), reps=5 if prec in ("fp64", "df64") else 20)
            c2.destroy()
            forms[prec] = {"matvec_ms": sec * 1e3, "matvec_tflops_fp64_equivalent": 6.0 * M * M * D / sec / 1e12,
                           "matvec_tflops_executed": 6.0 * M * M * D * TC_PRODUCTS[prec] / sec / 1e12}
        # whole solves of every form on the 63,000-unknown system (minutes in FP64 at n = 630,000)
        w2 = synth.workload(args.forms_workload)
        R2, y2 = torch.from_numpy(w2.R).to(dev), torch.from_numpy(w2.y).to(dev)
        forms_solve["workload"] = f"{w2.name}: n={w2.n}, {w2.select} k={w2.k}, lambda={w2.lam}"
        for prec in ("fp64", "df64", "ozaki", "tf32", "bf16"):
            torch.cuda.synchronize(dev)
            t0 = time.perf_counter()
            ph = step(prec, R2, y2, wl=w2)
            torch.cuda.synchronize(dev)
            ph["s"] = time.perf_counter() - t0
            ph["converged"] = ph["relres"] <= RTOL
            forms_solve[prec] = ph
        # the OZAKI form with a cheaper inner operator (6 and 5 of its 7 slice levels in the PCG
        # loop's matvec; FP64 true-residual restarts): "outer" counts the PCG runs
        for lev in (6, 5):
            torch.cuda.synchronize(dev)
            t0 = time.perf_counter()
            ph = step("ozaki", R2, y2, wl=w2, inner_levels=lev)
            torch.cuda.synchronize(dev)
            ph["s"] = time.perf_counter() - t0
            ph["converged"] = ph["relres"] <= RTOL
            forms_solve[f"ozaki_inner_levels_{lev}"] = ph

    cpu = None
    config1 = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cpu = cpu_baseline(w, head["iters"])
        config1 = config1_line(dev)

    if rank == 0:
        line = {
            "metric": METRIC, "value": t_dev, "unit": "s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": t_dev * 1e3, "higher_is_better": False, "scaling": "weak",
            "vs_baseline": None,
            "dtype": {"fp64": "f64", "df64": "f32x2 (double-float) contractions + f64",
                      "ozaki": "bf16 residues mod 14 numbers (exact FP32 sums) + f32x2 + f64", "tf32": "tf32 + f64",
                      "bf16": "bf16 + f64"}[args.precision], "data": "synthetic",
            "config": {"workload": f"{args.workload}: N={N} atoms, M={M} geometries, n={n}, D={D}, "
                                   f"{w.select} k={k}, sigma={w.sigma}, lambda={w.lam}, rtol={RTOL}",
                       "precision": args.precision, "select": w.select, "k": k, "n": n,
                       "parallelism": f"replicas x{world}",
                       "l2": "256 MB buffer written between timed steps (L2 129 MB); L_k working set "
                             f"{n * k * lbytes / 1e9:.2f} GB"},
            "solve": {"iters": head["iters"], "relres": head["relres"], "outer_steps": head["outer"],
                      "converged": head["relres"] <= RTOL, "setup_s": head["setup_s"], "build_s": head["build_s"],
                      "pcg_s": head["solve_s"], "s_per_iteration": head["solve_s"] / max(head["iters"], 1)},
            "e2e": {"value": t_e2e, "unit": "s", "h2d_bytes_per_step": int(R_h.numel() * 8 + y_h.numel() * 8),
                    "d2h_bytes_per_step": int(n * 8)},
            "roofline": roof_apply if ap_sec > mv_sec else roof_matvec,
            "roofline_matvec": roof_matvec,
            "roofline_apply": roof_apply,
            "cpu_baseline": cpu,
            "gpu_launches": int(launches),
            "clocks": clocks,
            "forms": forms,
            "forms_solve": forms_solve,
            "config1": config1,
        }
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()


# --------------------------------------------------------- CPU oracle arm
# PCG iterations of the headline (OZAKI) form on each workload, as the GPU arm measured them
# (its JSON line's solve.iters).  The FP64 oracle cannot run these solves to the end within a
# benchmark's time, so the reference arm extrapolates its sampled per-iteration cost with
# these counts; the GPU arm's own CPU baseline uses the iteration count of its run instead.
REF_ITERS = {"ethanol9_m200": 595, "aspirin21_m1000": 1578, "mol42_m5000": 3254}


def blas_info() -> dict:
    """BLAS library NumPy links and the thread settings of this process."""
    import numpy as np
    info = {"omp_num_threads": os.environ.get("OMP_NUM_THREADS"),
            "openblas_num_threads": os.environ.get("OPENBLAS_NUM_THREADS"), "nproc": os.cpu_count()}
    try:
        b = np.show_config(mode="dicts")["Build Dependencies"]["blas"]
        info["blas"] = f"{b.get('name')} {b.get('version')}"
    except Exception:  # older NumPy: no dict form
        info["blas"] = "unknown"
    return info


def _timed(fn):
    t = time.perf_counter()
    fn()
    return time.perf_counter() - t


def oracle_sample(w, iters: int) -> dict:
    """Time the FP64 oracle (as it stands) on bounded samples of one solve of workload w and
    extrapolate to the whole solve: setup-free preconditioner build + iters x (matvec + apply).

    Every term is a timing of the oracle's own functions, scaled by the size it was sampled at:
    * matvec: matvec_rows on 2 and 8 geometry blocks -> fixed + per-block cost, times M blocks;
    * Woodbury apply (Eq. 4) at the full k on two row panels of a random L_k -> fixed + per-row;
    * kernel columns (Eq. 5, Alg. 1): one column timed, times the columns the build takes;
    * dense k x k Cholesky timed at the full k; the n k^2 triangular solve and L^T L product
      timed on a row panel and scaled to n;
    * Algorithm 1 (pivoted Cholesky builds): 24 and 48 steps, fitted to a + b m per step.
    """
    import numpy as np
    import scipy.linalg as sla

    from oracle import kernel as ok
    from oracle import precond as op

    t0 = time.perf_counter()
    n, k, M = w.n, w.k, w.M
    rng = np.random.default_rng(0)
    v = rng.standard_normal(n)
    # matvec: fixed part (descriptors, Jacobians, W = J v) + one O(M D) pass per geometry block
    b1, b2 = min(M, 4), min(M, 24)
    ok.matvec_rows(w.R, w.sigma, v, [0], w.lam)  # first touch of the Jacobian's pages
    ta = _timed(lambda: ok.matvec_rows(w.R, w.sigma, v, list(range(b1)), w.lam))
    tb = _timed(lambda: ok.matvec_rows(w.R, w.sigma, v, list(range(b2)), w.lam))
    per_blk = max((tb - ta) / max(b2 - b1, 1), 0.0)
    t_mv = max(ta - b1 * per_blk, 0.0) + M * per_blk
    # Woodbury apply at the full k on row panels of n
    n1, n2 = min(n, 2000), min(n, 6000)
    LC = np.linalg.cholesky(w.lam * np.eye(k) + np.eye(k))
    t_ap_rows = []
    for rows in (n1, n2):
        Lk = rng.standard_normal((rows, k)) / np.sqrt(n)
        t_ap_rows.append(_timed(lambda: op.woodbury_apply(Lk, LC, w.lam, v[:rows])))
        del Lk
    per_row = max((t_ap_rows[1] - t_ap_rows[0]) / max(n2 - n1, 1), 0.0)
    t_ap = max(t_ap_rows[0] - n1 * per_row, 0.0) + n * per_row
    # dense pieces of the build at the full k, and the n k^2 products on a row panel
    A = rng.standard_normal((k, k)) / np.sqrt(k)
    A = A @ A.T + np.eye(k)
    t_chol = _timed(lambda: np.linalg.cholesky(A))
    Lkk = np.linalg.cholesky(A)
    ns = min(n, 600)
    Kp = rng.standard_normal((ns, k))
    t_trsm = _timed(lambda: sla.solve_triangular(Lkk, Kp.T, lower=True)) * n / ns
    t_syrk = _timed(lambda: Kp.T @ Kp) * n / ns
    del A, Lkk, Kp
    if w.select == "pivchol":
        get_col = ok.column_getter(w.R, w.sigma)
        d = ok.force_kernel_diag(w.R, w.sigma)
        m1 = 24
        T1 = _timed(lambda: op.pivoted_cholesky(get_col, d, m1))
        T2 = _timed(lambda: op.pivoted_cholesky(get_col, d, 2 * m1))
        b = max((T2 - 2 * T1) / (m1 * m1), 0.0)
        a = max((T1 - b * m1 * m1 / 2) / m1, 0.0)
        t_build = a * k + b * k * k / 2 + t_syrk + t_chol
        build_note = (f"Alg. 1 {m1} and {2 * m1} steps timed (a + b m per step), L^T L on {ns} rows, "
                      f"k x k Cholesky")
    else:
        # one kernel column costs one D x D Hessian block per geometry: timed on the first Ms
        # geometries of the workload and scaled to all M
        Ms = min(M, 400)
        get_sub = ok.column_getter(w.R[:Ms], w.sigma)
        get_sub(0)
        t_col = _timed(lambda: get_sub(1)) * M / Ms
        if w.select == "rls":  # pilot factor + its core + scores, then the final factor + core
            ncols, ntrsm, nsyrk, nchol = 2 * k, 3, 2, 4
        else:
            ncols, ntrsm, nsyrk, nchol = k, 1, 1, 2
        t_build = ncols * t_col + ntrsm * t_trsm + nsyrk * t_syrk + nchol * t_chol
        build_note = (f"1 kernel column ({t_col:.2f} s, timed on {Ms} of {M} geometries) x {ncols}, {ntrsm} "
                      f"triangular solves and {nsyrk} "
                      f"L^T L on {ns} of {n} rows, {nchol} k x k Cholesky at k={k}")
    total = t_build + iters * (t_mv + t_ap)
    return {"value": total, "unit": "s", "iters": iters, "build_s": t_build, "matvec_s": t_mv, "apply_s": t_ap,
            "sampled_s": time.perf_counter() - t0,
            "sample": (f"extrapolated from timed samples of workload {w.name}: matvec on {b1} and {b2} of {M} geometry "
                       f"blocks ({t_mv:.2f} s per matvec), Woodbury apply at k={k} on {n1} and {n2} of {n} rows "
                       f"({t_ap:.3f} s per apply), build: {build_note} ({t_build:.1f} s); total = build + {iters} "
                       f"PCG iterations x (matvec + apply)")}


def _sample_cmdline(workload: str, iters: int) -> list:
    return [sys.executable, os.path.abspath(__file__), "--cpu-sample", workload, "--ref-iters", str(iters)]


def config1_line(dev) -> dict:
    """The smallest system (ethanol9_m200: N = 9, M = 200, n = 5400, uniform k = 100,
    lambda = 1e-10): the GPU solve (setup, build, PCG to 1e-8) in FP64 and OZAKI against the
    paper's "analytic" baseline -- the oracle's dense K and Cholesky solve on the host, timed
    in full -- and the oracle's matrix-free PCG, timed on 30 iterations and scaled by the GPU's
    iteration count."""
    import numpy as np
    import torch

    from oracle import kernel as ok
    from oracle import precond as op
    from oracle import solver as osv
    from paper_2212_12737_gb300 import gdml, synth

    w = synth.workload("ethanol9_m200")
    R, y = torch.from_numpy(w.R).to(dev), torch.from_numpy(w.y).to(dev)
    out = {"workload": f"{w.name}: n={w.n}, {w.select} k={w.k}, lambda={w.lam}, rtol={RTOL}"}
    for prec in ("fp64", "ozaki"):
        best = None
        for _ in range(3):  # the first call captures the PCG graph
            torch.cuda.synchronize(dev)
            t0 = time.perf_counter()
            ctx = gdml.kernel_setup(R, w.sigma, w.lam, precision=prec)
            ctx.precond_build(w.select, w.k, seed=2)
            _, it, rel, _ = ctx.pcg_solve(y, rtol=RTOL, max_iter=20000, raise_on_nonconvergence=False)
            torch.cuda.synchronize(dev)
            t = time.perf_counter() - t0
            ctx.destroy()
            best = t if best is None else min(best, t)
        out[f"gpu_{prec}"] = {"s": best, "iters": it, "relres": rel}
    t0 = time.perf_counter()
    K = ok.force_kernel_dense(w.R, w.sigma)
    t1 = time.perf_counter()
    alpha = osv.solve_exact(K, w.lam, w.y)
    t2 = time.perf_counter()
    rel_cf = float(np.linalg.norm(w.y - K @ alpha - w.lam * alpha) / np.linalg.norm(w.y))
    S = op.select_uniform(w.n, w.k, 2)
    L, _ = op.nystrom_factor(K[:, S], S)
    LC = op.woodbury_core(L, w.lam)
    t3 = time.perf_counter()
    res = osv.pcg(lambda v: ok.matvec(w.R, w.sigma, v, w.lam), lambda r: op.woodbury_apply(L, LC, w.lam, r),
                  w.y, rtol=1e-30, max_iter=30, max_restarts=0)
    t4 = time.perf_counter()
    out["cpu_closed_form"] = {"s": t2 - t0, "assemble_K_s": t1 - t0, "cholesky_solve_s": t2 - t1,
                              "relres": rel_cf, "cores": os.cpu_count(), "kind": "oracle"}
    out["cpu_pcg_extrapolated"] = {"s": (t4 - t3) / res.iters * out["gpu_fp64"]["iters"],
                                   "sampled_iterations": res.iters, "per_iteration_s": (t4 - t3) / res.iters,
                                   "iters": out["gpu_fp64"]["iters"], "kind": "oracle", "extrapolated": True}
    return out


def cpu_baseline(w, gpu_iters: int) -> dict:
    """The oracle's extrapolated solve time on all host cores (this process) and on one core
    (a child process with every BLAS / OpenMP pool limited to one thread)."""
    allc = oracle_sample(w, gpu_iters)
    info = blas_info()
    env = dict(os.environ, OMP_NUM_THREADS="1", OPENBLAS_NUM_THREADS="1", MKL_NUM_THREADS="1")
    one = None
    try:
        out = subprocess.run(_sample_cmdline(w.name, gpu_iters), env=env, capture_output=True, text=True,
                             timeout=600)
        lines = [l for l in out.stdout.splitlines() if l.startswith("{")]
        one = json.loads(lines[-1]) if out.returncode == 0 and lines else None
    except (OSError, subprocess.TimeoutExpired, ValueError):
        one = None
    res = {"value": allc["value"], "unit": "s", "cores": info["nproc"], "kind": "oracle", "extrapolated": True,
           "sample": allc["sample"], "iters": gpu_iters, "build_s": allc["build_s"], "matvec_s": allc["matvec_s"],
           "apply_s": allc["apply_s"], "blas": info["blas"], "omp_num_threads": info["omp_num_threads"],
           "sampled_s": allc["sampled_s"]}
    if one:
        res["one_core"] = {"value": one["value"], "cores": 1, "build_s": one["build_s"],
                           "matvec_s": one["matvec_s"], "apply_s": one["apply_s"], "sampled_s": one["sampled_s"],
                           "env": "OMP_NUM_THREADS=OPENBLAS_NUM_THREADS=MKL_NUM_THREADS=1"}
    return res


def run_cpu_sample(args):
    """--cpu-sample: one oracle sample in this process, one JSON line (used for the 1-core run)."""
    from paper_2212_12737_gb300 import synth
    w = synth.workload(args.cpu_sample)
    out = oracle_sample(w, args.ref_iters or REF_ITERS.get(args.cpu_sample, 1000))
    out.update(blas_info())
    print(json.dumps(out), flush=True)


def run_reference(args):
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    from paper_2212_12737_gb300 import synth
    w = synth.workload(args.workload)
    iters = args.ref_iters or REF_ITERS[args.workload]
    vals = []
    info = None
    for i in range(args.warmup + args.steps):
        info = oracle_sample(w, iters)
        if i >= args.warmup:
            vals.append(info["value"])
    v = sum(vals) / len(vals)
    bi = blas_info()
    line = {"metric": METRIC, "value": v, "unit": "s", "impl": "reference", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": v * 1e3, "higher_is_better": False, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": args.workload, "precision": "fp64 (CPU oracle)", "select": w.select, "k": w.k,
                       "n": w.n},
            "extrapolated": True,
            "iters_source": ("the GPU arm's measured PCG iteration count for this workload (REF_ITERS in "
                             "bench.py, or --ref-iters); the oracle's own full solve does not fit a benchmark"),
            "cpu_baseline": {"value": v, "unit": "s", "cores": bi["nproc"], "kind": "oracle", "extrapolated": True,
                             "sample": info["sample"], "iters": iters, "blas": bi["blas"],
                             "omp_num_threads": bi["omp_num_threads"]},
            "e2e": {"value": v, "unit": "s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


if __name__ == "__main__":
    a = parse()
    if a.cpu_sample:
        run_cpu_sample(a)
    elif a.impl == "reference":
        run_reference(a)
    elif a.suite == "learned":
        run_learned(a)
    elif a.suite == "sym":
        run_sym(a)
    elif a.suite:
        run_suite(a)
    elif a.only != "solve":
        run_op(a)
    else:
        run_gpu(a)
