#!/usr/bin/env python3
"""Benchmark: all-eigenpair solve of the FP64 generalized eigenproblem A y = lambda B y
at M = 32768 (tight-binding pencil, 8192 atoms x 4 sp orbitals) on one GB300.

Contract (one JSON line on rank 0):
  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl gb300|reference]
A step is one full solve (Cholesky, reduction, tridiagonalisation, divide and conquer,
Householder back-transform, back-substitution) of a device-resident pencil;
`value` is seconds per solve (max over ranks).  Under torchrun every rank solves its
own pencil (replicas; the method has no exchange step).  --impl reference times the
FP64 CPU oracle on the machine's host cores on a bounded sample of the same workload.
"""
from __future__ import annotations

import argparse
import json
import math
import os
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "GEP solve time (all eigenpairs, FP64-accurate) at M=32768"


def parse():
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=1)
    p.add_argument("--warmup", type=int, default=3)
    p.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    p.add_argument("--M", type=int, default=32768)
    p.add_argument("--seed", type=int, default=0)
    p.add_argument("--precision", default="fp64_emulated", choices=["fp64_emulated", "fp64", "mixed_refined"])
    p.add_argument("--reducer", default="twosided", choices=["twosided", "explicit_inv", "eigenexa"],
                   help="reducer: two-sided (L^-1 never formed), explicit inverse, or the Cholesky-free "
                        "reducer of Eq. 7-9")
    p.add_argument("--sep", default="2stage", choices=["1stage", "2stage", "jacobi"],
                   help="SEP solver: 1-stage tridiagonalisation, full->band->tridiagonal, or block Jacobi")
    p.add_argument("--n-want", type=int, default=0,
                   help="only the lowest n eigenpairs (0: all; the occupied states are n = M/2)")
    p.add_argument("--bandwidth", type=int, default=0, help="band width of --sep 2stage (0: library default, 32 up to order 20480 and 64 beyond)")
    p.add_argument("--values-only", action="store_true", help="eigenvalues only (T_evo of the paper's benchmark)")
    p.add_argument("--cpu-sample-M", type=int, nargs="+", default=[1024, 2048, 3072],
                   help="orders of the oracle solves the c M^3 fit of the CPU baseline is taken over")
    p.add_argument("--profile-solve", action="store_true",
                   help="one untimed solve of the pencil with the given options and exit (profiling aid: "
                        "the command ncu launch lists and kernel captures of whole solves run)")
    p.add_argument("--peaks", action="store_true",
                   help="measure the FP64 peaks of this GPU (cuBLAS DGEMM burst and sustained) and exit")
    p.add_argument("--no-e2e", action="store_true")
    p.add_argument("--no-cpu", action="store_true")
    p.add_argument("--no-check", action="store_true")
    p.add_argument("--gemm-form", default="NNF", choices=["NNF", "NTL", "SNF"],
                   help="--gemm: transa, transb, uplo (NTL: lower rank-k update, SNF: symmetric A, k = m)")
    p.add_argument("--gemm", type=int, nargs=3, metavar=("m", "n", "k"),
                   help="time only the split-BF16 product engine on an m x n x k product (profiling aid)")
    p.add_argument("--compare-mixed", action="store_true",
                   help="mixed+refined vs FP64-accurate solve of the same pencil (default M=16384)")
    p.add_argument("--batched", action="store_true",
                   help="512 tight-binding pencils, orders log-uniform in [64, 2048], one captured graph")
    p.add_argument("--batch-count", type=int, default=512)
    p.add_argument("--nstreams", type=int, default=16, help="--batched: concurrent streams of the batch")
    p.add_argument("--batch-sep", default="auto", choices=["auto", "1stage", "2stage"],
                   help="--batched: SEP reduction of the pencils on the streams (auto: autotuned per bucket)")
    p.add_argument("--batch-small", type=int, default=-1,
                   help="--batched: order limit of the one-CTA route (-1: autotuned, 0: off, <= 128)")
    p.add_argument("--adjoint", action="store_true",
                   help="forward+adjoint of sum(lambda_occ) + <W, P> at M=4096 with central differences")
    p.add_argument("--fd-dirs", type=int, default=64)
    return p.parse_args()


def _median_clock(clk):
    return clk.stop()


def spectral_norm_lower_bound(A, iters=200, seed=0):
    """||A||_2 from below by power iteration (plain torch FP64): a conservative stand-in for
    the 2-norm in the |dlambda| <= 1e-11 ||A||_2 tolerance where a full eigensolve is too slow."""
    import torch
    g = torch.Generator(device="cpu").manual_seed(seed)
    v = torch.randn(A.shape[0], generator=g, dtype=torch.float64).to(A.device)
    v /= v.norm()
    lam = 0.0
    for _ in range(iters):
        u = A @ v
        lam = float(u.norm())
        v = u / lam
    return lam


def run_compare_mixed(a):
    """Config 3: the mixed-precision form (FP32-grade split-BF16 products, then FP64 refinement)
    against the plain FP64 form (every product on the FP64 units) and the FP64-accurate
    split-BF16 form, on the same pencil: wall time, stage times, and the error of the
    FP32-grade first pass alone and of the refined result, in |dlambda| / ||A||_2 against
    the FP64 forms, sampled residual and B-orthogonality."""
    import torch
    import gep_inputs as gi
    from paper_1504_06443_gb300 import build as gbuild
    import paper_1504_06443_gb300 as gep
    gbuild.build()
    M = a.M if a.M != 32768 else 16384
    tb = gi.tight_binding(M, a.seed)
    A = torch.as_tensor(tb["A"]).cuda()
    B = torch.as_tensor(tb["B"]).cuda()
    nA = spectral_norm_lower_bound(A)
    routes = [("fp64", "fp64", 0), ("fp64_emulated", "fp64_emulated", 0), ("mixed_refined", "mixed_refined", 0),
              ("mixed_first_pass", "mixed_refined", -1)]
    res, ws = {}, {}
    for name, prec, iters in routes:
        h = gep.Handle()
        steps = 1 if prec == "fp64" else a.steps
        for _ in range(max(1, a.warmup) if prec != "fp64" else 1):
            w, Y, info = gep.solve(A, B, precision=prec, timers=True, handle=h, sep=a.sep, refine_iters=iters)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(steps):
            w, Y, info = gep.solve(A, B, precision=prec, timers=True, handle=h, sep=a.sep, refine_iters=iters)
        e1.record()
        torch.cuda.synchronize()
        res[name] = {"s": e0.elapsed_time(e1) / steps / 1e3, "steps": steps, "info": info,
                     "stage_ms": [round(x, 1) for x in h.stage_times()],
                     "check": sampled_check(A, B, w, Y, 64, a.seed),
                     "refine_steps": h.refine_steps() if prec == "mixed_refined" else 0}
        ws[name] = w.clone()
        del Y
        h.close()
        torch.cuda.empty_cache()
    for name in res:
        res[name]["max_abs_dlambda_vs_fp64_over_normA"] = float((ws[name] - ws["fp64"]).abs().max()) / nA
        res[name]["max_abs_dlambda_vs_fp64_emulated_over_normA"] = float((ws[name] - ws["fp64_emulated"]).abs().max()) / nA
    out = {"metric": "mixed+refined vs FP64 GEP solve time at 1e-11 ||A||_2", "M": M, "unit": "s",
           "higher_is_better": False, "data": "synthetic", "dtype": "f64",
           "config": {"workload": f"tight-binding GEP M={M} ({M // 4} atoms), all eigenpairs", "sep": a.sep},
           "normA_2_lower_bound": nA, "normA_kind": "power iteration (200 steps), a lower bound of ||A||_2",
           "routes": res,
           "speedup_mixed_vs_fp64": res["fp64"]["s"] / res["mixed_refined"]["s"],
           "speedup_mixed_vs_fp64_emulated": res["fp64_emulated"]["s"] / res["mixed_refined"]["s"],
           "mixed_meets_1e-11": res["mixed_refined"]["max_abs_dlambda_vs_fp64_over_normA"] <= 1e-11}
    print(json.dumps(out), flush=True)


def run_batched(a):
    import time
    import torch
    import gep_inputs as gi
    from paper_1504_06443_gb300 import build as gbuild
    import paper_1504_06443_gb300 as gep
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    dist = None
    if world > 1:  # independent pencils: LPT shares, no exchange on the data path
        import torch.distributed as dist
        torch.cuda.set_device(int(os.environ.get("LOCAL_RANK", "0")))
        dist.init_process_group("nccl", device_id=torch.device("cuda", int(os.environ.get("LOCAL_RANK", "0"))))
    gbuild.build()
    all_orders = gi.batch_orders(a.batch_count, seed=1000)
    mine = gep.shard_batch(all_orders, world)[rank]
    orders = [all_orders[i] for i in mine]
    t0 = time.time()
    As, Bs = [], []
    for i, M in zip(mine, orders):
        tb = gi.tight_binding(M, 1000 + i)  # pencil i of the whole batch, whichever rank solves it
        As.append(torch.as_tensor(tb["A"]).cuda())
        Bs.append(torch.as_tensor(tb["B"]).cuda())
    gen_s = time.time() - t0
    reps = [next(i for i, M in enumerate(orders) if gep._bucket(M) == b) for b in sorted({gep._bucket(M) for M in orders})]
    tuner = gep.Autotuner()
    mixed = a.precision == "mixed_refined"
    # per size bucket the fastest route: engine (FP32-grade + FP64 refinement for every pencil
    # in the mixed form) x SEP reduction
    engines = ("mixed_refined",) if mixed else ("fp64", "fp64_emulated")
    tuner.tune([As[i] for i in reps], [Bs[i] for i in reps], reps=1, seps=("1stage",), engines=engines)
    precs = [tuner.precision_for(M) for M in orders]
    tuner.sep_threshold = 0  # the one-CTA choice is timed eagerly, with the few-launch 2-stage route
    small = tuner.tune_small(As, Bs, nstreams=a.nstreams, precision="mixed_refined" if mixed else None)
    if a.batch_sep == "auto":  # order above which pencils take the 2-stage route, timed on graphs
        tuner.tune_routes(As, Bs, nstreams=a.nstreams, precision="mixed_refined" if mixed else None)
    else:
        tuner.sep_threshold = None if a.batch_sep == "1stage" else 0
    sep_of = [tuner.sep_for(M) for M in orders] if a.batch_small < 0 else a.batch_small
    flops = sum(7.0 * float(M) ** 3 for M in orders)
    # looping single solves on one stream (baseline)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for A, B, p, sp in zip(As, Bs, precs, sep_of):
        gep.solve(A, B, precision=p, sep=sp)
    e1.record()
    torch.cuda.synchronize()
    loop_s = e0.elapsed_time(e1) / 1e3
    bs = gep.BatchedSolver(As, Bs, nstreams=a.nstreams, precisions=precs, seps=sep_of, batch_small=small)
    graph_note = "one captured CUDA graph"
    try:
        bs.capture()
        launch = bs.replay
    except ValueError as ex:  # too many kernels for one graph: the batch runs eagerly
        graph_note = f"none ({ex}); eager launches"
        launch = bs.run
    for _ in range(a.warmup):
        launch()
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    e0.record()
    for _ in range(a.steps):
        launch()
    e1.record()
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    s = e0.elapsed_time(e1) / a.steps / 1e3
    info = bs.info()
    if dist:
        t = torch.tensor([s, loop_s, float(info)], dtype=torch.float64, device="cuda")
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        s, loop_s, info = t[0].item(), t[1].item(), int(t[2].item())
        flops = sum(7.0 * float(M) ** 3 for M in all_orders)
    if rank != 0:
        if dist:
            dist.destroy_process_group()
        return
    orders = all_orders
    out = {"metric": "batched GEP throughput (all eigenpairs" + (", mixed+refined)" if mixed else ")"),
           "value": len(orders) / s, "unit": "GEPs/s", "gpu_launches": bs.graph_kernels or bs.eager_kernels,
           "n_gpus": world, "scaling": "strong" if world > 1 else None,
           "higher_is_better": True, "seconds_per_batch": s, "looping_single_solves_s": loop_s,
           "speedup_vs_loop": loop_s / s, "fp64_equiv_tflops": flops / s / 1e12, "info": info,
           "steps": a.steps, "warmup": a.warmup, "data": "synthetic", "dtype": "f64",
           "config": {"workload": f"{len(orders)} tight-binding pencils, M log-uniform in [64, 2048]",
                      "orders_min_max": [min(orders), max(orders)], "nstreams": a.nstreams, "graph": graph_note,
                      "autotuned_engine_per_bucket": {str(k): v for k, v in tuner.choice.items()},
                      "two_stage_above_order": tuner.sep_threshold,
                      "precision": "mixed_refined" if mixed else "FP64-accurate (engine per bucket)",
                      "one_cta_pencils_up_to": small,
                      "n_one_cta_pencils": sum(1 for M in orders if M <= small),
                      "generator_s": round(gen_s, 1),
                      "parallelism": f"LPT shards of the batch over {world} ranks" if world > 1 else "single"}}
    print(json.dumps(out), flush=True)
    if dist:
        dist.destroy_process_group()


def run_adjoint(a):
    import numpy as np
    import torch
    import gep_inputs as gi
    from paper_1504_06443_gb300 import build as gbuild
    import paper_1504_06443_gb300 as gep
    gbuild.build()
    M = a.M if a.M != 32768 else 4096
    n = M // 2
    tb = gi.tight_binding(M, a.seed)
    A = torch.as_tensor(tb["A"]).cuda().requires_grad_(True)
    B = torch.as_tensor(tb["B"]).cuda().requires_grad_(True)
    W = torch.as_tensor(gi.random_symmetric(M, 1)).cuda()

    def loss_of(A_, B_):
        w, P = gep.eigh_density(A_, B_, n)
        return w[:n].sum() + (W * P).sum(), w

    for _ in range(max(1, a.warmup)):
        loss, w = loss_of(A, B)
        gA, gB = torch.autograd.grad(loss, (A, B))
    torch.cuda.synchronize()
    e0, e1, e2 = (torch.cuda.Event(enable_timing=True) for _ in range(3))
    e0.record()
    loss, w = loss_of(A, B)
    e1.record()
    gA, gB = torch.autograd.grad(loss, (A, B))
    e2.record()
    torch.cuda.synchronize()
    gap = float((w[n] - w[n - 1]).item())
    rng = np.random.default_rng(2)
    h = 1e-6
    errs, errs2, errs_r = [], [], []
    with torch.no_grad():
        for _ in range(a.fd_dirs):
            dA = rng.standard_normal((M, M)); dA = dA + dA.T
            dB = rng.standard_normal((M, M)); dB = dB + dB.T
            dA *= 1e-3 * np.linalg.norm(tb["A"]) / np.linalg.norm(dA)
            dB *= 0.1 * 0.1 / np.linalg.norm(dB)
            dAt, dBt = torch.as_tensor(dA).cuda(), torch.as_tensor(dB).cuda()
            an = float((gA * dAt).sum() + (gB * dBt).sum())
            fd = {}
            for hh in (h, 2 * h):  # central differences at h and 2h (Richardson: O(h^4))
                fp, _ = loss_of(A + hh * dAt, B + hh * dBt)
                fm, _ = loss_of(A - hh * dAt, B - hh * dBt)
                fd[hh] = (fp - fm).item() / (2 * hh)
            rich = (4.0 * fd[h] - fd[2 * h]) / 3.0
            errs.append(abs(fd[h] - an) / max(1.0, abs(fd[h])))
            errs2.append(abs(fd[2 * h] - an) / max(1.0, abs(fd[2 * h])))
            errs_r.append(abs(rich - an) / max(1.0, abs(rich)))
    out = {"metric": "differentiable GEP: forward + adjoint time", "M": M, "n_occ": n, "unit": "s",
           "forward_s": e0.elapsed_time(e1) / 1e3, "backward_s": e1.elapsed_time(e2) / 1e3,
           "value": e0.elapsed_time(e2) / 1e3, "higher_is_better": False, "homo_lumo_gap": gap,
           "fd_directions": a.fd_dirs, "fd_h": h, "fd_max_rel_err": max(errs) if errs else None,
           "fd_median_rel_err": float(np.median(errs)) if errs else None,
           "fd_2h_max_rel_err": max(errs2) if errs2 else None,
           "fd_richardson_max_rel_err": max(errs_r) if errs_r else None,
           "data": "synthetic", "dtype": "f64",
           "config": {"workload": f"tight-binding GEP M={M}, loss = sum_occ lambda + <W, Y_o Y_o^T>"}}
    print(json.dumps(out), flush=True)


def run_gemm(a):
    """Engine-only timing (used for ncu captures of the product kernel on a small case)."""
    import torch
    from paper_1504_06443_gb300 import build as gbuild
    import paper_1504_06443_gb300 as gep
    gbuild.build()
    m, n, k = a.gemm
    ta, tb, uplo = a.gemm_form
    if ta == "S":
        k = m
    g = torch.Generator(device="cuda").manual_seed(a.seed)
    A = torch.randn(m, k, dtype=torch.float64, device="cuda", generator=g)
    B = torch.randn((n, k) if tb == "T" else (k, n), dtype=torch.float64, device="cuda", generator=g)
    C = torch.zeros((n, m), dtype=torch.float64, device="cuda").t()
    h = gep.default_handle()
    form = dict(transa=ta, transb=tb, uplo=uplo)
    for _ in range(a.warmup):
        gep.dgemm(A, B, engine=a.precision, C=C, handle=h, **form)
    torch.cuda.synchronize()
    h.profile_enable(4096)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(a.steps):
        gep.dgemm(A, B, engine=a.precision, C=C, handle=h, **form)
    e1.record()
    torch.cuda.synchronize()
    prof = h.profile_read()
    h.profile_enable(0)
    ms = e0.elapsed_time(e1) / a.steps
    useful = 2.0 * m * n * k * (0.5 if uplo == "L" else 1.0)
    print(json.dumps({"gemm": [m, n, k], "form": a.gemm_form, "engine": a.precision, "ms_per_call": ms,
                      "fp64_equiv_tflops": useful / (ms * 1e-3) / 1e12,
                      "kernel_ms_per_call": prof["ms"] / max(1, a.steps),
                      "kernel_tensor_tflops": prof["tensor_flops"] / (prof["ms"] * 1e-3) / 1e12 if prof["ms"] else None}),
          flush=True)


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f), "measured"
    except Exception:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0, "sm_max_mhz": 2070.0}, \
            "fallback"


class Clocks:
    """nvidia-smi sampler for the timed region."""

    FIELDS = "clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown," \
             "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown," \
             "clocks_event_reasons.sw_power_cap"

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                                          "-lms", "200", "-i", str(self.index)], stdout=subprocess.PIPE,
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
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [x.strip() for x in ln.split(",")]
            if len(parts) < 7:
                continue
            try:
                sm.append(float(parts[0]))
                mx = float(parts[1])
            except ValueError:
                continue
            for nm, v in zip(names, parts[3:7]):
                if v.lower() == "active":
                    reasons.add(nm)
        sm.sort()
        med = sm[len(sm) // 2] if sm else None
        return {"sm_mhz": med, "sm_max_mhz": mx, "reasons": sorted(reasons), "samples": len(sm)}


def cpu_sample(M_s, seed):
    """Oracle (FP64 CPU) full solve of an M_s tight-binding pencil; returns (seconds, cores, info)."""
    import gep_inputs as gi
    import oracle
    cores = os.cpu_count() or 1
    os.environ.setdefault("OMP_NUM_THREADS", str(cores))
    oracle.build()
    tb = gi.tight_binding(M_s, seed)
    t0 = time.perf_counter()
    _, _, info = oracle.gep_solve(tb["A"], tb["B"], want_vectors=True)
    dt = time.perf_counter() - t0
    return dt, int(os.environ.get("OMP_NUM_THREADS", cores)), info


def cm3_fit(samples, M):
    """Least-squares fit t = c M^3 over (M_s, seconds) samples, extrapolated to order M."""
    num = sum(t * float(m) ** 3 for m, t in samples)
    den = sum(float(m) ** 6 for m, _ in samples)
    c = num / den
    return c * float(M) ** 3, c


def cpu_baseline_fit(M, sizes, seed):
    """The oracle as it stands, timed on the host cores at several orders, with the c M^3
    fit extrapolated to order M (labelled as such)."""
    samples, cores = [], None
    for Ms in sizes:
        dt, cores, _ = cpu_sample(Ms, seed)
        samples.append((Ms, dt))
    v, c = cm3_fit(samples, M)
    return {"value": v, "unit": "s", "cores": cores, "kind": "oracle", "extrapolated": True,
            "fit": "t = c M^3, least squares", "c_s_per_M3": c,
            "samples_s": {str(m): round(t, 3) for m, t in samples},
            "sample": (f"oracle full GEP solves (all eigenpairs) of tight-binding pencils of order "
                       f"{', '.join(str(m) for m in sizes)} on {cores} host threads; the c M^3 fit is "
                       f"extrapolated to M={M}")}


def run_reference(a, rank, world):
    """The reference arm: there is no reference implementation of the method (a paper
    only), so the FP64 CPU oracle is timed as it stands.  Each step is one oracle solve of a
    bounded sample (orders rotating over --cpu-sample-M); the M = 32768 value is the c M^3 fit
    of the timed samples, labelled extrapolated."""
    if rank != 0:
        return
    M, sizes = a.M, list(a.cpu_sample_M)
    for _ in range(a.warmup):
        cpu_sample(min(sizes), a.seed)
    samples, cores = [], None
    t0 = time.perf_counter()
    for i in range(max(a.steps, len(sizes))):
        Ms = sizes[i % len(sizes)]
        dt, cores, info = cpu_sample(Ms, a.seed)
        samples.append((Ms, dt))
    wall = time.perf_counter() - t0
    v, c = cm3_fit(samples, M)
    sample = (f"{len(samples)} oracle full GEP solves (all eigenpairs) of tight-binding pencils of order "
              f"{', '.join(str(m) for m in sizes)} (rotating) on {cores} host threads; value = the c M^3 "
              f"least-squares fit extrapolated to M={M}")
    line = {"impl": "reference", "metric": METRIC, "value": v, "unit": "s", "n_gpus": world, "steps": len(samples),
            "warmup": a.warmup, "ms_per_step": v * 1e3, "higher_is_better": False, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic", "extrapolated": True,
            "sample_wall_s": round(wall, 2), "sample_ms_per_step": round(wall / len(samples) * 1e3, 1),
            "config": {"workload": f"tight-binding GEP M={M} ({M // 4} atoms x 4 sp orbitals), all eigenpairs",
                       "M": M, "seed": a.seed, "sampled_M": sizes},
            "cpu_baseline": {"value": v, "unit": "s", "cores": cores, "kind": "oracle", "extrapolated": True,
                             "c_s_per_M3": c, "sample": sample},
            "e2e": {"value": v, "unit": "s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def fp64_peaks(n=8192, burst_reps=5, sustained_s=3.0):
    """FP64 throughput of this GPU measured with cuBLAS DGEMM (torch.matmul on float64,
    2 n^3 flops per call): best of burst_reps calls, and back to back for sustained_s seconds.
    This is the FP64 tensor-core (DMMA) rate the paper's FP64 solvers would run at."""
    import torch
    a = torch.randn(n, n, dtype=torch.float64, device="cuda")
    b = torch.randn(n, n, dtype=torch.float64, device="cuda")
    c = a @ b
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = None
    for _ in range(burst_reps):
        e0.record()
        torch.matmul(a, b, out=c)
        e1.record()
        torch.cuda.synchronize()
        t = e0.elapsed_time(e1) / 1e3
        best = t if best is None or t < best else best
    reps = max(1, int(sustained_s / best))
    e0.record()
    for _ in range(reps):
        torch.matmul(a, b, out=c)
    e1.record()
    torch.cuda.synchronize()
    sus = e0.elapsed_time(e1) / 1e3 / reps
    f = 2.0 * n ** 3
    del a, b, c
    torch.cuda.empty_cache()
    return {"fp64_dgemm_tflops": f / best / 1e12, "fp64_dgemm_tflops_sustained": f / sus / 1e12,
            "how": f"cuBLAS DGEMM {n}^3 via torch.matmul (float64): best of {burst_reps} (burst) and "
                   f"{reps} back to back (sustained), CUDA events"}


def run_profile_solve(a):
    """One solve of the tight-binding pencil of order --M (seed --seed) with the bench's solver
    options, synchronised, nothing timed: the command ncu launch lists and kernel captures of a
    whole solve run."""
    import torch
    import gep_inputs as gi
    from paper_1504_06443_gb300 import build as gbuild
    import paper_1504_06443_gb300 as gep
    gbuild.build()
    tb = gi.tight_binding(a.M, a.seed)
    A = torch.as_tensor(tb["A"], device="cuda")
    B = torch.as_tensor(tb["B"], device="cuda")
    w, Y, info = gep.solve(A, B, reducer=a.reducer, sep=a.sep, bandwidth=a.bandwidth, precision=a.precision,
                           want_vectors=not a.values_only, timers=True)
    torch.cuda.synchronize()
    print(json.dumps({"profile_solve": a.M, "info": info, "stage_ms": [round(x, 2) for x in
                                                                       gep.default_handle().stage_times()]}))


def run_peaks(a):
    import torch
    torch.cuda.set_device(int(os.environ.get("LOCAL_RANK", "0")))
    out = fp64_peaks()
    out["gpu"] = torch.cuda.get_device_name()
    print(json.dumps(out), flush=True)


# DRAM traffic of one launch of each product kernel from ncu captures (dram__bytes_read.sum +
# dram__bytes_write.sum).  They are scaled to the timed launches by their tensor flops (36 and 16 plane products per FP64 product) and reported only
# while the kernel sources are the ones that were captured.
PRODUCT_CAPTURES = {
    "digits": {"dram_bytes": 2.225633e9 + 0.169617e9, "tensor_flops": 36 * 2.0 * 4096 ** 3, "planes": 36,
               "source": "gemm_oz.cu", "from": "template <int SC, int LC, int TNC = TN>", "to": "size_t smem_bytes_for",
               "kernel_sha1": "12e778370d0c233aad0046fed42ad573ed9f796c"},
    "residues": {"dram_bytes": 0.802419e9 + 0.109109e9, "tensor_flops": 16 * 2.0 * 4096 * 2048 * 4096, "planes": 16,
                 "source": "gemm_res.cu", "from": "__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(RTHREADS",
                 "to": "// ------------------------------------------------------------------ reconstruction",
                 "kernel_sha1": "8bbf5a52937995625464c284537cdaa1e8861dd0"}}
TRAFFIC_NOTE = ("ncu dram__bytes_read.sum + dram__bytes_write.sum of one 4096^3 k_oz_gemm launch and one 4096 x 2048 x 4096 "
                "k_res_gemm launch, scaled to the average timed launch by its tensor flops; null when a kernel source "
                "differs from the captured one")


def product_kernel_sha1(c):
    """sha1 of a product kernel's source text, so that a capture of another version is not reported."""
    import hashlib
    path = os.path.join(ROOT, "paper_1504_06443_gb300", "csrc", c["source"])
    try:
        src = open(path).read()
        i = src.index(c["from"])
        j = src.index(c["to"], i)
        return hashlib.sha1(src[i:j].encode()).hexdigest()
    except (OSError, ValueError):
        return None


def product_traffic(prof):
    if not prof["launches"] or any(c["kernel_sha1"] != product_kernel_sha1(c) for c in PRODUCT_CAPTURES.values()):
        return None
    d, r = PRODUCT_CAPTURES["digits"], PRODUCT_CAPTURES["residues"]
    # the launches' FP64 flops by form, from their total and the tensor flops they took
    digits = max(prof["tensor_flops"] - r["planes"] * prof["fp64_flops"], 0.0) / (d["planes"] - r["planes"])
    residues = prof["fp64_flops"] - digits
    total = sum(c["dram_bytes"] * c["planes"] * f / c["tensor_flops"] for c, f in ((d, digits), (r, residues)))
    return total / prof["launches"]


STAGE_NAMES = ["R1_cholesky", "R2_reduce", "S1_tridiag", "S2_dc", "S3_back_q", "R3_backsub", "MP3_refine"]
# the Cholesky-free reducer (Eq. 7-9) records its own stages in the reducer's timer slots
STAGE_NAMES_EIGENEXA = ["E7_sep_of_B", "E8_A_prime", "S1_tridiag", "S2_dc", "S3_back_q", "E9_Y_is_XZ", "MP3_refine"]


def stage_names(reducer):
    return STAGE_NAMES_EIGENEXA if reducer == "eigenexa" else STAGE_NAMES


def stage_rooflines(M, stages, band_ms, vectors, sep, b, bf16_peak, f64pk, reducer="twosided", n=None):
    """Per-stage algorithmic FP64-equivalent flops (the method's counts, not the work the GPU
    path does) over the stage's CUDA-event time, against the measured FP64 DGEMM rate and, in
    terms of the 36 BF16 plane products one FP64-accurate product costs, against the measured
    sustained BF16 rate.  n < M: only the lowest n eigenpairs (back-transforms of n columns)."""
    m3 = float(M) ** 3
    n = M if n is None else n
    fr = float(n) / M
    back = (4.0 if sep == "2stage" else 2.0) * m3
    sep_alg = {"S1_tridiag": 4.0 / 3 * m3, "S2_dc": 4.0 / 3 * m3 if vectors else 0.0,
               "S3_back_q": back * fr if vectors else 0.0}
    if sep == "jacobi":  # one sweep's rotations, the least the block-Jacobi route can do
        sep_alg = {"S1_tridiag": 0.0, "S2_dc": 8.0 * m3, "S3_back_q": 0.0}
    if reducer == "eigenexa":
        sep_b = 4.0 / 3 * m3 + 4.0 / 3 * m3 + back if sep != "jacobi" else 8.0 * m3
        alg = {"E7_sep_of_B": sep_b, "E8_A_prime": 3.0 * m3, **sep_alg,
               "E9_Y_is_XZ": 2.0 * m3 * fr if vectors else 0.0, "MP3_refine": 0.0}
    else:
        alg = {"R1_cholesky": m3 / 3, "R2_reduce": m3, **sep_alg,
               "R3_backsub": m3 * fr if vectors else 0.0, "MP3_refine": 0.0}
    names = stage_names(reducer)
    f64 = f64pk.get("fp64_dgemm_tflops_sustained") if isinstance(f64pk, dict) else None
    out = {}

    def row(ms, flops, tensor=True):
        r = {"ms": round(ms, 2), "alg_flops": flops}
        if ms > 0 and flops > 0:
            tf = flops / (ms * 1e-3) / 1e12
            r["fp64_equiv_tflops"] = tf
            if f64:
                r["frac_of_fp64_dgemm"] = tf / f64
            if tensor and bf16_peak:
                # digits take 36 plane products per FP64 product (above 1 where the deep products' 16 residues do)
                r["frac_of_bf16_sustained_36_planes"] = tf * 36 / bf16_peak
                r["frac_of_bf16_sustained_16_planes"] = tf * 16 / bf16_peak
        return r

    for nm, t in zip(names, stages):
        if alg[nm] > 0:
            out[nm] = row(t, alg[nm])
    if band_ms:
        out["S1b_full_to_band"] = row(band_ms[0], 4.0 / 3 * m3)
        out["S1c_bulge_chasing"] = row(band_ms[1], 6.0 * b * float(M) ** 2, tensor=False)
    out["R1+R2_reducer"] = row(stages[0] + stages[1], alg[names[0]] + alg[names[1]])
    total = sum(alg.values()) + (6.0 * b * float(M) ** 2 if band_ms else 0.0)
    return {"stages": out, "whole_solve_alg_flops": total}


def sampled_check(A, B, w, Y, ncols=64, seed=0):
    """Residual / B-orthogonality / Rayleigh-quotient checks on sampled eigenpairs
    (plain torch FP64 on the GPU, independent of the solver library)."""
    import torch
    M, n = A.shape[0], Y.shape[1]
    ncols = min(ncols, n)
    g = torch.Generator(device="cpu").manual_seed(seed)
    idx = torch.randperm(n, generator=g)[:ncols].sort().values.to(A.device)
    Ys = Y[:, idx].contiguous()
    AY = A @ Ys
    BY = B @ Ys
    ws = w[idx]
    R = AY - BY * ws[None, :]
    res = (R.norm(dim=0) / (A.norm() / math.sqrt(M))).max().item()  # per-column, scaled like ||A||_F / sqrt(M)
    G = Ys.t() @ BY
    orth = (G - torch.eye(ncols, dtype=G.dtype, device=G.device)).abs().max().item()
    rq = ((Ys * AY).sum(0) / (Ys * BY).sum(0) - ws).abs().max().item()
    # ||A Y - B Y Lambda||_F / (||A||_F M), estimated from the sampled columns
    res_ns = math.sqrt(n / ncols * float((R * R).sum().item())) / (A.norm().item() * M)
    return {"cols": ncols, "residual_F_over_normF_M_est": res_ns, "max_col_residual_over_normA_rms": res,
            "orth_max": orth, "rayleigh_minus_w_max": rq, "ascending": bool((w[1:] >= w[:-1]).all().item())}


def main():
    a = parse()
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if a.peaks:
        run_peaks(a)
        return
    if a.profile_solve:
        run_profile_solve(a)
        return
    if a.gemm:
        run_gemm(a)
        return
    if a.compare_mixed:
        run_compare_mixed(a)
        return
    if a.batched:
        run_batched(a)
        return
    if a.adjoint:
        run_adjoint(a)
        return
    if a.impl == "reference":
        if world > 1:
            import torch.distributed as dist
            dist.init_process_group("gloo")
        run_reference(a, rank, world)
        return

    import numpy as np
    import torch
    import gep_inputs as gi
    from paper_1504_06443_gb300 import build as gbuild
    import paper_1504_06443_gb300 as gep

    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    gbuild.build()
    M = a.M
    seed = a.seed + rank
    t0 = time.time()
    tb = gi.tight_binding(M, seed)
    gen_s = time.time() - t0
    A = torch.as_tensor(tb["A"]).to("cuda")
    B = torch.as_tensor(tb["B"]).to("cuda")
    if a.no_e2e:
        del tb
    vectors = not a.values_only
    if not 0 <= a.n_want <= M:
        raise SystemExit(f"--n-want must lie in [0, {M}]")
    n = a.n_want or M
    sopts = dict(reducer=a.reducer, sep=a.sep, bandwidth=a.bandwidth, precision=a.precision, want_vectors=vectors,
                 n_want=a.n_want)
    w = torch.empty(n, dtype=torch.float64, device="cuda")
    Yt = torch.empty((n, M), dtype=torch.float64, device="cuda") if vectors else None
    h = gep.default_handle()
    opts = gep.make_options(timers=True, **sopts)
    h.ensure_workspace(gep.workspace_bytes(M, handle=h, timers=True, **sopts))
    stream = torch.cuda.current_stream()

    for _ in range(a.warmup):
        gep.solve_async(A, B, w, Yt, opts, h)
    torch.cuda.synchronize()
    info = h.info()
    # product-kernel launches per step (one untimed solve with per-launch events), so that the
    # events of the timed region cover every product launch of every timed step
    h.profile_enable(1 << 20)
    gep.solve_async(A, B, w, Yt, opts, h)
    per_step_products = h.profile_read(reset=True)["launches"]
    h.profile_enable(per_step_products * a.steps + 64)
    h.launches(reset=True)
    clk = Clocks(local)
    clk.start()
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(a.steps):
        gep.solve_async(A, B, w, Yt, opts, h)
    e1.record(stream)
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    clocks = clk.stop()
    ms = e0.elapsed_time(e1) / a.steps
    launches = h.launches(reset=True) / a.steps
    prof = h.profile_read(reset=True)
    h.profile_enable(0)
    stages = h.stage_times()
    band_ms = h.band_times() if a.sep == "2stage" else None
    info = max(info, h.info())
    t_local = torch.tensor([ms], dtype=torch.float64, device="cuda")
    if dist:
        dist.all_reduce(t_local, op=dist.ReduceOp.MAX)
    ms_max = t_local.item()

    check = None
    if not a.no_check and vectors:
        check = sampled_check(A, B, w, Yt.t(), 64, seed)

    e2e = None
    if not a.no_e2e:
        Ah = torch.from_numpy(tb["A"]).pin_memory()
        Bh = torch.from_numpy(tb["B"]).pin_memory()
        del tb
        wh = torch.empty(n, dtype=torch.float64).pin_memory()
        Yh = torch.empty((n, M), dtype=torch.float64).pin_memory() if vectors else None
        del Yt
        torch.cuda.empty_cache()
        hh = gep.Handle()
        import ctypes
        o = gep.make_options(**sopts)
        nb = ctypes.c_size_t()
        hh.lib.gep_workspace_size_host(hh.h, M, ctypes.byref(o), ctypes.byref(nb))
        h.ws = None
        torch.cuda.empty_cache()
        hh.ensure_workspace(nb.value)
        P = ctypes.c_void_p
        torch.cuda.synchronize()
        t1 = time.perf_counter()
        rc = hh.lib.gep_solve_host(hh.h, M, P(Ah.data_ptr()), M, P(Bh.data_ptr()), M, P(wh.data_ptr()),
                                   P(Yh.data_ptr() if vectors else 0), M, ctypes.byref(o))
        e2e_s = time.perf_counter() - t1
        e2e = {"value": e2e_s, "unit": "s", "h2d_bytes_per_step": 2 * 8 * M * M,
               "d2h_bytes_per_step": 8 * n + (8 * n * M if vectors else 0),
               "rc": rc, "max_abs_dw_vs_device": float((wh.cuda() - w).abs().max().item())}

    pk, pk_kind = peaks()
    try:
        f64pk = fp64_peaks(8192, burst_reps=3, sustained_s=2.0)
    except Exception as ex:  # the bench line stays valid without it
        f64pk = {"error": str(ex)}
    covered_steps = prof["launches"] / per_step_products if per_step_products else 0
    t_kernel_ms = prof["ms"] / covered_steps if covered_steps else None
    achieved = (prof["tensor_flops"] / (prof["ms"] * 1e-3) / 1e12) if prof["ms"] > 0 else None
    peak = pk.get("bf16_tflops_sustained", pk.get("bf16_tflops"))
    roof = {"bound": "tensor", "kernel": "k_oz_gemm and k_res_gemm (BF16 tcgen05 plane products)",
            "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
            "frac": (achieved / peak) if achieved else None,
            "traffic": product_traffic(prof),
            "traffic_note": TRAFFIC_NOTE,
            "peak_kind": f"{pk_kind} bf16 dense sustained",
            "fp64_equiv_tflops": (prof["fp64_flops"] / (prof["ms"] * 1e-3) / 1e12) if prof["ms"] > 0 else None,
            "kernel_ms_per_step": t_kernel_ms, "timed_launches": prof["launches"], "untimed_launches": prof["skipped"],
            "launches_per_step": per_step_products, "steps_covered": covered_steps,
            "share_of_step": (t_kernel_ms / ms) if t_kernel_ms else None}

    bw = (a.bandwidth or (32 if a.M <= 20480 else 64)) if a.sep == "2stage" else 0
    stage_roof = stage_rooflines(M, stages, band_ms, vectors, a.sep, bw, peak, f64pk, reducer=a.reducer, n=n)

    # the CPU baseline is the oracle's full solve (all eigenpairs), the default workflow's work
    full_workflow = vectors and n == M and a.reducer != "eigenexa"
    cpu = None
    if rank == 0 and world == 1 and not a.no_cpu and full_workflow:
        del A, B
        torch.cuda.empty_cache()
        cpu = cpu_baseline_fit(M, list(a.cpu_sample_M), a.seed)

    flops_alg = stage_roof["whole_solve_alg_flops"]
    if rank == 0:
        what = ("all eigenvalues" if not vectors else "all eigenpairs" if n == M
                else f"lowest {n} eigenpairs")
        metric = METRIC if (vectors and n == M) else f"GEP solve time ({what}, FP64-accurate) at M={M}"
        line = {"metric": metric, "value": ms_max / 1e3, "unit": "s", "n_gpus": world, "steps": a.steps,
                "warmup": a.warmup, "ms_per_step": ms_max, "higher_is_better": False, "scaling": "weak",
                "vs_baseline": None, "dtype": "f64", "data": "synthetic",
                "config": {"workload": f"tight-binding GEP M={M} ({M // 4} atoms x 4 sp orbitals), " + what,
                           "n_want": a.n_want,
                           "M": M, "seed": a.seed, "reducer": a.reducer, "sep": a.sep,
                           "bandwidth": (a.bandwidth or (32 if a.M <= 20480 else 64)) if a.sep == "2stage" else None,
                           "precision": a.precision, "parallelism": "replicas" if world > 1 else "single",
                           "l2": (f"inputs larger than L2 ({8.0 * M * M / 1e9:.2f} GB per matrix, L2 129 MB)"
                                  if 8.0 * M * M > 129e6 else
                                  f"inputs smaller than L2 ({8.0 * M * M / 1e6:.1f} MB per matrix), not flushed"),
                           "generator_s": round(gen_s, 2)},
                "stage_ms": dict(zip(stage_names(a.reducer), [round(x, 2) for x in stages])),
                "band_ms": dict(zip(["S1b_full_to_band", "S1c_bulge_chasing"], [round(x, 2) for x in band_ms]))
                if band_ms else None,
                "info": info, "gpu_launches": int(launches),
                "fp64_equiv_tflops_whole_solve": flops_alg / (ms_max * 1e-3) / 1e12,
                "roofline": roof, "stage_roofline": stage_roof["stages"], "fp64_peak": f64pk,
                "clocks": clocks, "e2e": e2e, "cpu_baseline": cpu, "check": check}
        print(json.dumps(line), flush=True)
    if dist:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
