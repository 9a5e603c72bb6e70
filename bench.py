#!/usr/bin/env python
"""Benchmark of the overlap operator's hot path on GB300.

Metric: sgn(gamma5 D_w(mu)) b solves/s at 1e-8 relative error, the mixed
precision batched form (the headline) next to the FP64 form, the single-source
forms and Arnoldi, plus the Wilson stencil's bandwidth against the HBM roof.

Workload (one step = one batch): the 12 spin-colour point sources at site 0 on
each of four lattices of uneven sizes, 6^4, 8^4, 12^4 and 16^3 x 8 (48
sequences, 58896 sites), SU(3) links U = exp(i eps H) with eps = 1.0 (seeds
1003-1006), m_w = -1.5 (kappa = 0.2), mu = 0.2, antiperiodic time, the 20
eigenvalues of A nearest the imaginary axis deflated on each lattice (left/right
eigenvectors from the library's GPU eigensolver, set-up untimed); every source
gives D_ov(mu) b = b + gamma5 sgn(A) b.  The Krylov size k is the smallest on a
grid for which every source agrees to 1e-8 with a self-converged FP64 solve
(k = 1500) and the sources the FP64 oracle reaches (6^4 and 8^4; stored by
tests/golden/make_oracle_refs.py) agree with the oracle to 1e-8.  Inputs are
resident in HBM when the timed region starts; L2 is flushed (a 512 MiB write)
before every timed step and each step is timed on the device with CUDA events.
Extras (context, not the headline): the same batch in FP64, 16^3 x 8 with 30
deflated eigenpairs in single-source mixed precision, a batch of 12 Gaussian
sources on 8^4 (mu = 0.3), single-source and Arnoldi solves on 8^4, the
gradients and the stencil bandwidth on 48^3 x 64.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

N > 1 runs under torchrun: each rank solves its own batch on its own GPU
(replicas; the path has no data exchange), the max over ranks of the timed
device time sets the aggregate rate.  --impl reference times the FP64 CPU
oracle (scipy sparse matvec + numpy) on a bounded sample of the same workload,
one process per host core.
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

METRIC = "sgn(γ5Dw(μ))b solves/s at 1e-8 rel err, mixed vs FP64; Dw GB/s vs HBM peak"
# headline: 12 point sources on each of four lattices of uneven sizes, one batch per step
HEAD_DIMS = [(6, 6, 6, 6), (8, 8, 8, 8), (12, 12, 12, 12), (16, 16, 16, 8)]
HEAD_SEEDS = [1003, 1004, 1005, 1006]
HEAD_MU, HEAD_M = 0.2, 20
HEAD_K_GRID = list(range(400, 1001, 10))
HEAD_K_REF = 1500
# Krylov size of the reference arm (the driver runs it before this arm, so it cannot read this
# arm's calibration): the k the calibration below chose on GB300 for the headline batch
REF_K_DEFAULT = 480
HEAD_WORKLOAD = ("12 spin-colour point sources x 4 lattices {6^4, 8^4, 12^4, 16^3x8} (48 sequences, "
                 "58896 sites), SU(3) exp(i*1.0*H) links, m_w=-1.5, mu=0.2, batched two-sided Lanczos, "
                 "20 eigenvalues of smallest |Re lambda| deflated per lattice")
ORACLE_REFS = os.path.join(ROOT, "tests", "golden", "oracle_refs.npz")
# the 8^4 Gaussian-source batch (an extra)
DIMS = (8, 8, 8, 8)
EPS, SEED_U, SEED_B = 1.0, 1001, 2001
MU, KAPPA = 0.3, 0.2
K_GRID = list(range(300, 1001, 10))
K_REF = 1000
RS_M, RS_MAX_CYCLES = 60, 24  # restarted Arnoldi extra: steps per cycle (fastest of 40-200 at 8^4), most cycles
OV_NEV = 6  # eigenvalues of D_ov nearest 0 in the 8^4 extras
DW_DIMS = (48, 48, 48, 64)  # 7.1M sites: every stencil operand is far larger than L2
LARGE_K = 40  # Krylov steps of the single-source timing on that lattice (cost per step)
NRHS = 12
WORKLOAD8 = ("8^4 lattice (N=49152), SU(3) exp(i*1.0*H) links, m_w=-1.5, mu=0.3, batches of 12 Gaussian b, "
             "two-sided Lanczos, 20 eigenvalues of smallest |Re lambda| deflated")
# config of 16^3 x 8 with 30 deflated eigenpairs (an extra): single-source mixed precision
C3_DIMS, C3_SEED_U, C3_SEED_B, C3_MU, C3_M = (16, 16, 16, 8), 1002, 2002, 0.3, 30
# dram__bytes_read.sum + dram__bytes_write.sum per launch of the headline batch's dominant kernel
# class, from one ncu capture of the current kernels (the roofline's "traffic"); None until measured
HEAD_TRAFFIC = {"pass2_batched_doublefloat": 836263168}  # k_b_regen_df, 48 sequences, one launch
# ncu dram__bytes_read + write per launch of the single stencil on 48^3 x 64 (row-grouped block order;
# profiles/stencil_dslash_48x48x48x64_and_32x32x32x64.md)
DW_TRAFFIC = {"f32_12": 2.970e9, "f32_18": 3.625e9, "f64": 9.75e9}


def peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return d.get("hbm_gbs", 6800.0), "measured"
    return 6800.0, "fallback"


# FP64 ALU roof: 152 SMs x 2 FP64 FMA / clock / SM x 2 flop x 2.07 GHz = 1.259 TFLOP/s
FP64_PEAK_TFLOPS = 152 * 2 * 2 * 2.07e9 / 1e12
# algorithmic work per site: Wilson hopping term 1320 flop, diagonal and
# gamma5 48 flop; FP64 bytes: 4 links (576) + x (192) + y (192)
DW_FLOP_SITE = 1368
DW_BYTES = {"f64": 960, "f32_12": 384, "f32_18": 480}
# two-pass regeneration step (FP64): stencil + recurrence/accumulate epilogue of 12 complex
REGEN_FLOP_SITE = DW_FLOP_SITE + 12 * 30
REGEN_BYTES_SITE = 576 + 192 + 192 + 2 * 192 + 192
# fused FP32 pass-1 step (pair stencil + 2sL recurrence): 12-real links (192) + v_i, w_i (192) +
# v_{i-1}, w_{i-1} (192) + write v_{i+1}, w_{i+1} (192); t, s stay on chip
PASS1_BYTES_SITE = 768
# FP32 operations (add, multiply or fused multiply-add: one each) of one double-float regeneration
# step per site, counted from the arithmetic of df32.cuh in the kernel: per hop the projection
# (12 unnormalised double-float sums x 8), the link product (6 complex outputs x 134: one exact
# product of 4 operations and 11 compensated terms of 12, two renormalisations of 3), the
# coefficient (13 double-float products x 7); per output component the hop sum (16 x 8), the real
# 1/beta_i times a complex number (2 x 7), three complex double-float products (50 each) and three
# complex sums (22 each)
REGEN_DF_OPS_SITE = 8 * (12 * 8 + 6 * 134 + 13 * 7) + 12 * (16 * 8 + 2 * 7 + 3 * 50 + 3 * 22)
# the same step as k_b_regen_df evaluates it (kappa folded into the step's coefficients, sums of products
# renormalised once): per hop 12 sums of 8, 12 sums of 6 products at 64, 24 spin sums of 8; 168 for the
# temporal coefficients; per part of an output component 52 + 30 and three renormalisations of 3
REGEN_DFX_OPS_SITE = 8 * (12 * 8 + 12 * 64 + 24 * 8) + 168 + 24 * (52 + 30 + 3 * 3)
# FP32 issue rate: 152 SMs x 128 lanes x 2.07 GHz (one operation per lane and clock)
FP32_OPS_PEAK_T = 152 * 128 * 2.07e9 / 1e12
# FP64 pass-2 step: links (576) + v_i (192) + v_{i-1} (192) + v_{i+1} write (192) + y read/write (384)
PASS2_BYTES_SITE = 1536
M_DEFL = 20


def kernel_roofline(name, ms_per_launch, steps, V, hbm_peak):
    """Algorithmic work of one launch of a kernel class divided by its measured duration."""
    if name == "pass1_persistent":
        return {"bound": "hbm", "achieved": PASS1_BYTES_SITE * V * steps / ms_per_launch / 1e6, "peak": hbm_peak,
                "unit": "GB/s", "algorithmic": f"{PASS1_BYTES_SITE} B/site/step x {V} sites x {steps} steps"}
    if name == "pass2_persistent":
        return {"bound": "alu", "achieved": REGEN_FLOP_SITE * V * steps / ms_per_launch / 1e9,
                "peak": FP64_PEAK_TFLOPS, "unit": "TFLOP/s",
                "algorithmic": f"{REGEN_FLOP_SITE} FP64 flop/site/step x {V} sites x {steps} steps"}
    if name == "dslash_regen":
        return {"bound": "alu", "achieved": REGEN_FLOP_SITE * V / ms_per_launch / 1e9, "peak": FP64_PEAK_TFLOPS,
                "unit": "TFLOP/s", "algorithmic": f"{REGEN_FLOP_SITE} FP64 flop/site x {V} sites"}
    if name == "dslash_pair":
        return {"bound": "hbm", "achieved": (2 * 96 * 2 + 192) * V / ms_per_launch / 1e6, "peak": hbm_peak,
                "unit": "GB/s", "algorithmic": f"576 B/site x {V} sites"}
    return None


class Clocks:
    """nvidia-smi samples (200 ms) during the timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.Q}", "--format=csv,noheader,nounits",
                 "-lms", "200"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except Exception:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if not self.proc:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx = float(f[2])
            except ValueError:
                continue
            for nm, v in zip(names, f[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": mx,
                "reasons": sorted(reasons), "samples": len(sm)}


def max_over_ranks(x: float, world: int, device) -> float:
    """The largest x over the ranks of the job (the timing rule: the slowest replica sets the rate)."""
    if world == 1:
        return x
    import torch
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_rate(total_ms_max: float, world: int, units_per_step: int, steps: int) -> float:
    """Units solved by all replicas per second of the slowest replica's timed device time."""
    return world * units_per_step * steps / (total_ms_max / 1e3)


def dist_setup():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def calibrate_k(ovl, ctx, torch, b, flags_list, grid=None, oref=None):
    """Smallest k on K_GRID whose solve agrees with the FP64 k=1000 solve to 1e-8 (and, given the
    oracle's stored reference of b, with the oracle to 1e-8 as well); entries of flags_list are
    (name, flags) for two-sided Lanczos or (name, flags, method)."""
    ref, _ = ctx.sign_krylov(ovl.LANCZOS2, K_REF, MU, KAPPA, b)
    ref = ref.clone()
    nrm = torch.linalg.vector_norm(ref).item()
    out = {}
    for entry in flags_list:
        name, fl = entry[0], entry[1]
        method = entry[2] if len(entry) > 2 else ovl.LANCZOS2
        kg = grid or K_GRID
        chosen, err = kg[-1], None
        for k in kg:
            y, info = ctx.sign_krylov(method, k, MU, KAPPA, b, flags=fl)
            e = torch.linalg.vector_norm(y - ref).item() / nrm
            eo = None
            if oref is not None and e <= 1e-8:
                d = oracle_error(y, oref)
                eo = max(d["sampled_rel"], d["proj_rel"])
            print(f"[bench] calibrate {name} k={k} err={e:.3e} err_oracle={eo}", file=sys.stderr, flush=True)
            if e <= 1e-8 and (eo is None or eo <= 1e-8):
                chosen, err = k, e
                break
            err = e
        out[name] = (chosen, err)
    return out


def time_solves(torch, ctx, fn, bufs, warmup, steps, flush):
    """Per-step device time (CUDA events on the library's stream), L2 flushed before each step."""
    st = torch.cuda.current_stream()
    times = []
    for i in range(warmup + steps):
        flush.fill_(i)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(st)
        fn(bufs[i % len(bufs)])
        e1.record(st)
        e1.synchronize()
        if i >= warmup:
            times.append(e0.elapsed_time(e1))
    return times


def large_single_source(torch, ovl, ctx, k=LARGE_K):
    """One Gaussian source on the stencil lattice, mixed two-sided Lanczos at a fixed k (the cost
    per Krylov step, not a converged solve): the default path (on a lattice above the persistent
    limit, the batched kernels as a batch of one, double-float regeneration) against the stepwise
    single-source kernels (FP64 regeneration), each against the FP64 two-pass solve of the same k.
    The lattice is far larger than L2, so no flush is needed between solves."""
    b = torch.randn(ctx.n, dtype=torch.complex128, device="cuda", generator=torch.Generator("cuda").manual_seed(7))
    y = torch.empty_like(b)
    st = torch.cuda.current_stream()
    out = {"k": k, "mu": MU}
    y64 = ctx.sign_krylov(ovl.LANCZOS2, k, MU, KAPPA, b, flags=ovl.TWO_PASS)[0].clone()
    for name, fl in (("default_batch_of_one", ovl.MIXED), ("stepwise", ovl.MIXED | ovl.STEPWISE)):
        ctx.sign_krylov(ovl.LANCZOS2, k, MU, KAPPA, b, y, flags=fl)  # tuning, graph capture
        ts = []
        for _ in range(3):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(st)
            ctx.sign_krylov(ovl.LANCZOS2, k, MU, KAPPA, b, y, flags=fl)
            e1.record(st)
            e1.synchronize()
            ts.append(e0.elapsed_time(e1))
        err = (torch.linalg.vector_norm(y - y64) / torch.linalg.vector_norm(y64)).item()
        out[name] = {"ms": round(statistics.median(ts), 2), "rel_vs_fp64_two_pass": err}
    del b, y, y64
    return out


def dw_bandwidth(torch, ovl, reps=20, dims=DW_DIMS, single_source=None):
    """Stencil GB/s on a lattice far larger than L2 (device-layout vectors).  With a dict for
    single_source, also the single-source solve timing of large_single_source on that lattice."""
    from paper_0810_4228_gb300 import synth
    V = dims[0] * dims[1] * dims[2] * dims[3]
    ctx = ovl.Context(dims)
    U = synth.gauge_field_torch(dims, EPS, SEED_U, device="cuda")
    ctx.set_gauge(U)
    del U
    torch.cuda.empty_cache()
    res = {}
    st = torch.cuda.current_stream()
    for name, flag, prec in (("f32_12", ovl.F32, 1), ("f32_18", ovl.F32_FULL, 1), ("f64", 0, 0)):
        x = ctx.empty_native(prec)
        if prec == 1:
            x.copy_(torch.randn(ctx.n, dtype=torch.complex64, device="cuda"))
        else:
            x.copy_(torch.randn(ctx.n, dtype=torch.complex128, device="cuda"))
        y = ctx.empty_native(prec)
        for _ in range(3):
            ctx.apply_Dw(MU, KAPPA, x, y, flags=ovl.GAMMA5 | ovl.NATIVE | flag)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(st)
        for _ in range(reps):
            ctx.apply_Dw(MU, KAPPA, x, y, flags=ovl.GAMMA5 | ovl.NATIVE | flag)
        e1.record(st)
        e1.synchronize()
        ms = e0.elapsed_time(e1) / reps
        res[name] = {"ms": ms, "GB_s": DW_BYTES[name] * V / ms / 1e6, "GFLOP_s": DW_FLOP_SITE * V / ms / 1e6}
        if name == "f32_12":
            # the fused pair t = A v, s = A^dag w with alpha = w^dag t (12-real links read once for both:
            # 576 B/site); each call ends with the host read of alpha, which the timing includes
            w = ctx.empty_native(1)
            w.copy_(torch.randn(ctx.n, dtype=torch.complex64, device="cuda"))
            t, s = ctx.empty_native(1), ctx.empty_native(1)
            for _ in range(3):
                ctx.apply_pair(MU, KAPPA, x, w, t, s, prec=1)
            e0.record(st)
            for _ in range(reps):
                ctx.apply_pair(MU, KAPPA, x, w, t, s, prec=1)
            e1.record(st)
            e1.synchronize()
            msp = e0.elapsed_time(e1) / reps
            res["pair_f32_12"] = {"ms": msp, "GB_s": 576 * V / msp / 1e6, "GFLOP_s": 2 * DW_FLOP_SITE * V / msp / 1e6}
            del w, t, s
        del x, y
    torch.cuda.empty_cache()
    if single_source is not None:
        try:
            single_source.update(large_single_source(torch, ovl, ctx))
        except Exception as exc:  # report, keep the stencil measurement
            single_source["error"] = repr(exc)[:200]
    ctx.close()
    torch.cuda.empty_cache()
    return dims, V, res


def _oracle_worker(task):
    """One host process of the oracle sample: the oracle's two-sided Lanczos recurrence from one
    point source of one headline lattice for a bounded number of steps (single-threaded)."""
    j, r, budget_s, k = task
    for v in ("OPENBLAS_NUM_THREADS", "OMP_NUM_THREADS", "MKL_NUM_THREADS"):
        os.environ[v] = "1"
    if ROOT not in sys.path:
        sys.path.insert(0, ROOT)
    import numpy as np
    from oracle import krylov as K
    from oracle import wilson as W
    from paper_0810_4228_gb300 import synth
    dims = HEAD_DIMS[j]
    U = synth.gauge_field(dims, EPS, HEAD_SEEDS[j])
    A = W.a_operator(U, dims, HEAD_MU, KAPPA)
    Ah = A.conj().T.tocsr()
    b = synth.point_sources(dims, site=0)[r]
    t0 = time.perf_counter()
    K.lanczos2(A.dot, Ah.dot, b, b, 4)
    t4 = (time.perf_counter() - t0) / 4
    s = int(max(8, min(k, budget_s / max(t4, 1e-9))))
    t0 = time.perf_counter()
    _, _, a_, be, ga = K.lanczos2(A.dot, Ah.dot, b, b, s)
    t_step = (time.perf_counter() - t0) / s
    # the inner sign at the full size: the oracle's dense sgn(G_k) e_1 of a k x k tridiagonal
    # (its cost does not depend on the values; the sample's coefficients, repeated)
    t_in = None
    if r == 0:
        def rep(x, n):
            return np.tile(x, -(-n // len(x)))[:n]
        t0 = time.perf_counter()
        K.inner_sign_e1(K.tridiag(rep(a_, k), rep(be, k - 1), rep(ga, k - 1)))
        t_in = time.perf_counter() - t0
    return {"j": j, "steps": s, "t_step": t_step, "t_inner": t_in}


def oracle_batch_sample(k: int, budget_s: float = 20.0, procs: int = 0):
    """The FP64 oracle on a bounded sample of the headline batch, on all host cores: one process
    per core (spawned), each running the oracle's two-sided Lanczos recurrence from a point source
    of one of the four lattices for about budget_s seconds; the per-step times measured under full
    load, with the oracle's dense inner sign at size k, give the time of the whole batch
    (12 sources x 4 lattices x (k steps + inner sign)) spread over the processes.  The deflation
    set-up is excluded (as on the GPU and in the paper); the deflation split of each source
    (a few dozen vector operations against k steps of two matvecs) is not timed."""
    import multiprocessing as mp
    P = max(procs or os.cpu_count() or 1, len(HEAD_DIMS))  # at least one process per lattice
    tasks = [(w % len(HEAD_DIMS), 0 if w < len(HEAD_DIMS) else (w // len(HEAD_DIMS)) % 12, budget_s, k)
             for w in range(P)]
    ctx = mp.get_context("spawn")
    t0 = time.perf_counter()
    with ctx.Pool(P) as pool:
        res = pool.map(_oracle_worker, tasks, chunksize=1)
    wall = time.perf_counter() - t0
    per_lat = {}
    for d in res:
        per_lat.setdefault(d["j"], []).append(d["t_step"])
    t_step = {j: statistics.median(v) for j, v in per_lat.items()}
    t_in = {d["j"]: d["t_inner"] for d in res if d["t_inner"] is not None}
    cpu_s = sum(NRHS * (k * t_step[j] + t_in[j]) for j in range(len(HEAD_DIMS)))
    batch_wall = cpu_s / P
    nseq = NRHS * len(HEAD_DIMS)
    return {"value": nseq / batch_wall, "unit": "solves/s", "cores": P, "kind": "oracle",
            "batch_seconds": batch_wall, "k": k, "sample_wall_s": round(wall, 1),
            "sample": (f"{P} concurrent single-threaded processes (one per host core) each ran "
                       f"{min(d['steps'] for d in res)}-{max(d['steps'] for d in res)} steps of the FP64 oracle's "
                       f"two-sided Lanczos (scipy CSR matvec + numpy) from a point source of one of the four "
                       f"lattices; per-step s under full load "
                       + ", ".join(f"{'x'.join(map(str, HEAD_DIMS[j]))}: {t_step[j]*1e3:.1f} ms" for j in sorted(t_step))
                       + f"; dense inner sign at k={k}: "
                       + ", ".join(f"{t_in[j]:.2f} s" for j in sorted(t_in))
                       + f"; batch = 12 sources x 4 lattices x (k steps + inner sign) / {P} processes")}


def run_reference(args, world, rank):
    if rank != 0:
        return
    k = args.k or REF_K_DEFAULT
    nrun = args.warmup + args.steps
    budget = max(4.0, min(20.0, 150.0 / max(nrun, 1)))
    t_all, last = [], None
    for i in range(nrun):
        last = oracle_batch_sample(k, budget_s=budget)
        if i >= args.warmup:
            t_all.append(last["batch_seconds"])
    per = sum(t_all) / len(t_all)
    nseq = NRHS * len(HEAD_DIMS)
    val = nseq / per
    line = {"metric": METRIC, "value": val, "unit": "solves/s", "n_gpus": args.gpus, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": per * 1e3, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": HEAD_WORKLOAD, "dims": [list(d) for d in HEAD_DIMS], "mu": HEAD_MU,
                       "kappa": KAPPA, "eps": EPS, "k": k, "rhs_per_lattice": NRHS, "m_deflated": HEAD_M},
            "impl": "reference",
            "cpu_baseline": {"value": val, "unit": "solves/s", "cores": last["cores"], "kind": "oracle",
                             "sample": last["sample"]},
            "e2e": {"value": val, "unit": "solves/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line))


def batch_launches(nseq, k, m, persistent_pass1=True, fused_start=False):
    """Kernels one mixed batched solve launches: per sequence pack, state init, projections (two
    two-stage kernels), split, two FP32 conversions, the Newton fallback (two, they return at once
    when the quadrature settled), start vector, two and one double-float conversions, unpack; then
    pass 1 (one persistent launch, or pair + recurrence per step), the inner sign (prep, six levels
    of solve + sum) and k - 1 regeneration steps.  755 for 12 sequences, k = 550, m = 20 (the ncu
    launch list of one solve counts the same).  fused_start: the regeneration's start vectors, their
    conversions and the way back in one launch each for all sequences, plus one for the step
    coefficients, and the first two quadrature levels' solves in one launch, as the library does it now."""
    per_seq = 1 + 1 + (4 if m > 0 else 0) + 1 + 2 + 2 + 1 + 2 + 1 + 1
    pass1 = 1 if persistent_pass1 else 2 * k - 1
    if fused_start:
        return nseq * (per_seq - 4) + pass1 + 1 + 2 * 6 - 1 + 3 + (k - 1)
    return nseq * per_seq + pass1 + 1 + 2 * 6 + (k - 1)


def calibrate_batch(torch, bt, srcs, refs, flags, grid):
    """Smallest k on the grid for which every source of the batch is within 1e-8 of its reference."""
    chosen, err = grid[-1], None
    for k in grid:
        outs, _, _ = bt.solve(k, MU, KAPPA, [srcs], flags=flags)
        e = max(torch.linalg.vector_norm(outs[0][r] - refs[r]).item() / torch.linalg.vector_norm(refs[r]).item()
                for r in range(refs.shape[0]))
        print(f"[bench] calibrate batch flags={flags} k={k} err={e:.3e}", file=sys.stderr, flush=True)
        err = e
        if e <= 1e-8:
            chosen = k
            break
    return chosen, err


# row a10: per site of ovl_dw_grad, algorithmic bytes (x 192 + g 192 read, the link force
# 36 complex = 576 written, the temporal link 144 read for d/dmu) and FP64 operations counted
# from the kernel (per link two hops of two half-spinor projections, 24, and 18 complex
# multiply-adds of the colour outer products, 144, and their scaled sum, 36; the d/dmu term 72)
DWGRAD_BYTES_SITE = 192 + 192 + 576 + 144
DWGRAD_FLOP_SITE = 4 * (2 * (24 + 144) + 36) + 72


def autograd_timing(torch, ovl, U_np, b, flush, k=800, gdims=(24, 24, 24, 24)):
    """Row a10 on the GPU.  ovl_sign_grad (derivatives of Re <g, sgn(A) b> with respect to the links,
    mu and b, resolvent form: one FP64 two-sided Lanczos process from (b, g)) on the 8^4 workload at
    k = 800 (where the 8^4 gradient test meets central differences to 1e-5), against the FP64
    forward solve at the same k; ovl_dw_grad (adjoint of y = A x: link force and d/dmu) on a lattice
    far larger than L2.  CUDA events on the library's stream around each call (each call ends with
    its own host synchronisation, included).  Failures are reported, not raised."""
    from paper_0810_4228_gb300 import synth
    out = {}

    def timed(fn, reps):
        st = torch.cuda.current_stream()
        ts = []
        for i in range(reps + 1):  # the first call warms up
            flush.fill_(i & 0xFF)
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(st)
            fn()
            e1.record(st)
            e1.synchronize()
            ts.append(e0.elapsed_time(e1))
        return statistics.median(ts[1:])

    try:
        lat = ovl.Context(DIMS)
        lat.set_gauge(torch.from_numpy(U_np).cuda())
        g = torch.from_numpy(synth.gaussian_source(DIMS, SEED_B + 600)).cuda()
        bb = b.clone()
        gU = torch.empty((lat.V, 4, 3, 3), dtype=torch.complex128, device="cuda")
        gb, y = torch.empty_like(bb), torch.empty_like(bb)
        t_grad = timed(lambda: lat.sign_grad(k, MU, KAPPA, bb, g, y=y, grad_U=gU, grad_b=gb), 3)
        gm64 = lat.sign_grad(k, MU, KAPPA, bb, g, y=y, grad_U=gU, grad_b=gb)[0]
        gU64, gb64 = gU.clone(), gb.clone()
        t_mix = timed(lambda: lat.sign_grad(k, MU, KAPPA, bb, g, y=y, grad_U=gU, grad_b=gb, flags=ovl.MIXED), 3)
        gmm = lat.sign_grad(k, MU, KAPPA, bb, g, y=y, grad_U=gU, grad_b=gb, flags=ovl.MIXED)[0]
        t_fwd = timed(lambda: lat.sign_krylov(ovl.LANCZOS2, k, MU, KAPPA, bb, y), 3)

        def rel(a, r):
            return (torch.linalg.vector_norm(a - r) / torch.linalg.vector_norm(r)).item()
        out["sign_grad_8x4"] = {"k": k, "ms": round(t_grad, 3), "forward_fp64_ms": round(t_fwd, 3),
                                "ratio_to_forward": round(t_grad / t_fwd, 2),
                                "outputs": "sgn(A) b, grad_U, grad_mu, grad_b",
                                "mixed": {"ms": round(t_mix, 3), "ratio_to_forward": round(t_mix / t_fwd, 2),
                                          "rel_diff_vs_fp64": {"grad_U": rel(gU, gU64), "grad_b": rel(gb, gb64),
                                                               "grad_mu": abs(gmm - gm64) / abs(gm64)},
                                          "form": "FP32 Lanczos, double-float combination"}}
        lat.close()
        del gU, gb, y, g, bb, gU64, gb64
    except Exception as exc:  # report, keep the rest of the line
        out["sign_grad_8x4"] = {"error": repr(exc)[:200]}
    try:
        V2 = gdims[0] * gdims[1] * gdims[2] * gdims[3]
        lat2 = ovl.Context(gdims)
        U2 = synth.gauge_field_torch(gdims, EPS, SEED_U + 7, device="cuda")
        lat2.set_gauge(U2)
        del U2
        x = torch.randn(V2 * 12, dtype=torch.complex128, device="cuda")
        gg = torch.randn(V2 * 12, dtype=torch.complex128, device="cuda")
        gU2 = torch.empty((V2, 4, 3, 3), dtype=torch.complex128, device="cuda")
        ms = timed(lambda: lat2.dw_grad(MU, KAPPA, x, gg, gU2), 10)
        ms32 = timed(lambda: lat2.dw_grad(MU, KAPPA, x, gg, gU2, flags=ovl.F32), 10)
        out["dw_grad"] = {"dims": list(gdims), "sites": V2, "ms": round(ms, 4), "ms_f32": round(ms32, 4),
                          "GB_s": round(DWGRAD_BYTES_SITE * V2 / ms / 1e6, 1),
                          "GFLOP_s": round(DWGRAD_FLOP_SITE * V2 / ms / 1e6, 1),
                          "frac_fp64_roof": round(DWGRAD_FLOP_SITE * V2 / ms / 1e9 / FP64_PEAK_TFLOPS, 3),
                          "bytes_per_site": DWGRAD_BYTES_SITE, "flop_per_site": DWGRAD_FLOP_SITE,
                          "bound": "FP64 ALU (3.2 flop/B against 0.19 at the FP64 roof)"}
        lat2.close()
        del x, gg, gU2
        torch.cuda.empty_cache()
    except Exception as exc:  # report, keep the rest of the line
        out["dw_grad"] = {"error": repr(exc)[:200]}
    return out


def load_oracle_refs():
    """{case: {key: array}} from tests/golden/oracle_refs.npz (values written by the oracle), or {}."""
    if not os.path.exists(ORACLE_REFS):
        return {}
    import numpy as np
    z = np.load(ORACLE_REFS)
    out = {}
    for key in z.files:
        case, field = key.split("/", 1)
        out.setdefault(case, {})[field] = z[key]
    return out


_PROJ_CACHE = {}


def oracle_error(y, ref):
    """Distance of a full sgn(A) b vector y (torch or numpy) to the oracle's stored one: relative
    2-norm over the sampled components, their largest difference relative to their largest
    magnitude, and the relative error estimated from the eight stored projections
    g_j^dag sgn(A) b (E|g^dag e|^2 = 2 |e|^2: g has N(0, 1) real and imaginary parts)."""
    import numpy as np
    from paper_0810_4228_gb300 import synth
    yy = y.detach().cpu().numpy() if hasattr(y, "detach") else np.asarray(y)
    dims = tuple(int(d) for d in ref["dims"])
    if dims not in _PROJ_CACHE:
        _PROJ_CACHE[dims] = np.stack([synth.gaussian_source(dims, 9000 + j) for j in range(len(ref["proj"]))])
    G = _PROJ_CACHE[dims]
    d = yy[ref["idx"]] - ref["val"]
    pe = G.conj() @ yy - ref["proj"]
    return {"sampled_rel": float(np.linalg.norm(d) / np.linalg.norm(ref["val"])),
            "sampled_maxabs_rel": float(np.abs(d).max() / np.abs(ref["val"]).max()),
            "proj_rel": float(np.sqrt(np.mean(np.abs(pe) ** 2) / 2.0) / float(ref["norm"]))}


def headline_setup(torch, ovl, m=HEAD_M):
    """Contexts of the four lattices (fields drawn on the host: the oracle sees the same links),
    their deflation eigenpairs (library eigensolver, untimed) and the 12 point sources each."""
    from paper_0810_4228_gb300 import synth
    ctxs, srcs, setup = [], [], []
    for d, seed in zip(HEAD_DIMS, HEAD_SEEDS):
        c = ovl.Context(d)
        c.set_gauge(torch.from_numpy(synth.gauge_field(d, EPS, seed)).cuda())
        t0 = time.perf_counter()
        e = c.deflation_eigs(HEAD_MU, KAPPA, m) if m > 0 else {"m": 0, "max_residual": 0.0}
        setup.append({"dims": list(d), "m": e["m"], "seconds": round(time.perf_counter() - t0, 2),
                      "max_residual": e["max_residual"]})
        ctxs.append(c)
        srcs.append(torch.from_numpy(synth.point_sources(d, site=0)).cuda())
    return ctxs, srcs, setup


def headline_errors(torch, outs, refs64, orefs):
    """Largest relative error of the batch's sgn(A) b over all sources against the FP64 k = 1500
    solves, and over the oracle's sources (6^4, 8^4) against the oracle."""
    e64 = max(torch.linalg.vector_norm(outs[j][r] - refs64[j][r]).item() / torch.linalg.vector_norm(refs64[j][r]).item()
              for j in range(len(HEAD_DIMS)) for r in range(NRHS))
    eo = None
    for name, ref in orefs.items():
        j = [tuple(d) for d in HEAD_DIMS].index(tuple(int(x) for x in ref["dims"]))
        r = int(ref["source_arg"])
        e = oracle_error(outs[j][r], ref)
        v = max(e["sampled_rel"], e["proj_rel"])
        eo = v if eo is None else max(eo, v)
    return e64, eo


def calibrate_headline(torch, ovl, bt, ctxs, srcs, orefs, flags, grid):
    """Smallest k on the grid for which every source of the batch is within 1e-8 of its FP64
    k = 1500 solve and the oracle's sources are within 1e-8 of the oracle."""
    refs64 = [torch.stack([c.sign_krylov(ovl.LANCZOS2, HEAD_K_REF, HEAD_MU, KAPPA, srcs[j][r])[0].clone()
                           for r in range(NRHS)]) for j, c in enumerate(ctxs)]
    # the self-converged FP64 reference itself against the oracle
    ref_vs_oracle = None
    for name, ref in orefs.items():
        j = [tuple(d) for d in HEAD_DIMS].index(tuple(int(x) for x in ref["dims"]))
        e = oracle_error(refs64[j][int(ref["source_arg"])], ref)
        v = max(e["sampled_rel"], e["proj_rel"])
        ref_vs_oracle = v if ref_vs_oracle is None else max(ref_vs_oracle, v)
    chosen, e64, eo = grid[-1], None, None
    for k in grid:
        outs, _, _ = bt.solve(k, HEAD_MU, KAPPA, srcs, flags=flags)
        e64, eo = headline_errors(torch, outs, refs64, orefs)
        print(f"[bench] calibrate headline flags={flags} k={k} err_fp64={e64:.3e} err_oracle={eo}",
              file=sys.stderr, flush=True)
        if e64 <= 1e-8 and (eo is None or eo <= 1e-8):
            chosen = k
            break
    return chosen, e64, eo, ref_vs_oracle, refs64


def headline_launches(k, m=HEAD_M, fused_start=False):
    """Kernels one headline batch launches (batch_launches with the pass-1 form the batch takes:
    the 48 sequences' 128-site blocks exceed what one resident grid holds, so pass 1 runs stepwise)."""
    blocks = sum(NRHS * -(-(d[0] * d[1] * d[2] * d[3]) // 128) for d in HEAD_DIMS)
    return batch_launches(NRHS * len(HEAD_DIMS), k, m, persistent_pass1=blocks <= 3 * 152, fused_start=fused_start)


def gauss8_extras(torch, ovl, args, flush, orefs, hbm_peak, rank):
    """The 8^4 workload with Gaussian sources (mu = 0.3, 20 deflated): a batch of 12 sources, single
    sources (two-sided Lanczos mixed / FP64, Arnoldi FP64 / double-float), each at its calibrated k
    (1e-8 against the FP64 k = 1000 solve), the FP64 reference and the solves against the oracle's
    stored sgn(A) b of the source with seed 2001."""
    from paper_0810_4228_gb300 import synth
    U = synth.gauge_field(DIMS, EPS, SEED_U)
    srcs = torch.from_numpy(synth.gaussian_source(DIMS, SEED_B + 7919 * rank, nrhs=NRHS)).cuda()
    b1 = torch.from_numpy(synth.gaussian_source(DIMS, SEED_B)).cuda()  # the oracle's source
    ctx = ovl.Context(DIMS)
    ctx.set_gauge(torch.from_numpy(U).cuda())
    t0 = time.perf_counter()
    eig = ctx.deflation_eigs(MU, KAPPA, args.m) if args.m > 0 else None
    if eig:
        eig["seconds"] = round(time.perf_counter() - t0, 2)
    bt = ovl.Batch([ctx], [NRHS])
    fl_mix, fl_64 = ovl.MIXED | ovl.OVERLAP, ovl.OVERLAP
    oref = orefs.get("gauss8_mu0.3")
    refs = torch.stack([ctx.sign_krylov(ovl.LANCZOS2, K_REF, MU, KAPPA, srcs[r])[0].clone() for r in range(NRHS)])
    k_mix, err_mix = calibrate_batch(torch, bt, srcs, refs, ovl.MIXED, K_GRID)
    k_64, err_64 = calibrate_batch(torch, bt, srcs, refs, 0, K_GRID)
    cal = calibrate_k(ovl, ctx, torch, b1, [("mixed", ovl.MIXED), ("fp64", 0)], oref=oref)
    (k_s, err_s), (k_s64, err_s64) = cal["mixed"], cal["fp64"]
    cal_a = calibrate_k(ovl, ctx, torch, b1, [("arnoldi", 0, ovl.ARNOLDI), ("arnoldi_df", ovl.MIXED, ovl.ARNOLDI)],
                        grid=list(range(250, 801, 10)), oref=oref)
    (k_arn, err_arn), (k_adf, err_adf) = cal_a["arnoldi"], cal_a["arnoldi_df"]
    vs_oracle = None
    if oref is not None:
        vs_oracle = {}
        for name, meth, k, fl in (("fp64_k1000_reference", ovl.LANCZOS2, K_REF, 0),
                                  ("lanczos2_mixed", ovl.LANCZOS2, k_s, ovl.MIXED),
                                  ("lanczos2_fp64", ovl.LANCZOS2, k_s64, 0),
                                  ("arnoldi_fp64", ovl.ARNOLDI, k_arn, 0),
                                  ("arnoldi_doublefloat", ovl.ARNOLDI, k_adf, ovl.MIXED)):
            y = ctx.sign_krylov(meth, k, MU, KAPPA, b1, flags=fl)[0]
            vs_oracle[name] = dict(k=k, **oracle_error(y, oref))
    nctx = max(3, min(args.steps, 5))
    outb = torch.empty_like(srcs)
    t_b = time_solves(torch, ctx, lambda _: bt.solve(k_mix, MU, KAPPA, [srcs], [outb], flags=fl_mix), [0], 2, nctx,
                      flush)
    t_b64 = time_solves(torch, ctx, lambda _: bt.solve(k_64, MU, KAPPA, [srcs], [outb], flags=fl_64), [0], 2, nctx,
                        flush)
    out1 = torch.empty_like(srcs[0])
    bsingle = [srcs[r] for r in range(NRHS)]
    t_s = time_solves(torch, ctx, lambda b: ctx.sign_krylov(ovl.LANCZOS2, k_s, MU, KAPPA, b, out1, flags=fl_mix),
                      bsingle, 2, nctx, flush)
    t_s64 = time_solves(torch, ctx, lambda b: ctx.sign_krylov(ovl.LANCZOS2, k_s64, MU, KAPPA, b, out1, flags=fl_64),
                        bsingle, 2, nctx, flush)
    single_profile, reproj = None, None
    try:
        ctx.profile(reset=True)
        ctx.sign_krylov(ovl.LANCZOS2, k_s, MU, KAPPA, srcs[0], out1, flags=fl_mix | ovl.PROFILE)
        torch.cuda.synchronize()
        single_profile = {kk: round(v["ms"], 4) for kk, v in ctx.profile(reset=True).items() if v.get("launches")}
    except Exception as exc:  # report, keep the rest of the line
        single_profile = {"error": repr(exc)[:200]}
    try:
        t_rp = time_solves(torch, ctx, lambda b: ctx.sign_krylov(ovl.LANCZOS2, k_s, MU, KAPPA, b, out1,
                                                                 flags=fl_mix | ovl.REPROJ), bsingle, 2, nctx, flush)
        reproj = {"k": k_s, "ms": round(statistics.mean(t_rp), 3), "ms_without": round(statistics.mean(t_s), 3),
                  "m": args.m}
        yr = ctx.sign_krylov(ovl.LANCZOS2, k_s, MU, KAPPA, srcs[0], flags=ovl.MIXED | ovl.REPROJ)[0]
        reproj["rel_err_vs_k1000_fp64"] = (torch.linalg.vector_norm(yr - refs[0]) /
                                           torch.linalg.vector_norm(refs[0])).item()
    except Exception as exc:  # report, keep the rest of the line
        reproj = {"error": repr(exc)[:200]}
    t_arn = time_solves(torch, ctx, lambda b: ctx.sign_krylov(ovl.ARNOLDI, k_arn, MU, KAPPA, b, out1,
                                                              flags=ovl.OVERLAP), bsingle, 1, 2, flush)
    t_adf = time_solves(torch, ctx, lambda b: ctx.sign_krylov(ovl.ARNOLDI, k_adf, MU, KAPPA, b, out1,
                                                              flags=ovl.OVERLAP | ovl.MIXED), bsingle, 2, nctx, flush)
    # the double-float Gram-Schmidt sweeps against HBM: the delayed CGS2 reads v_0..v_j twice at
    # step j (the classical form four times), 16 B per complex element (CUDA events around each
    # sweep kernel, eager launches)
    ctx.profile(reset=True)
    ctx.sign_krylov(ovl.ARNOLDI, k_adf, MU, KAPPA, srcs[0], out1, flags=ovl.OVERLAP | ovl.MIXED | ovl.PROFILE)
    torch.cuda.synchronize()
    aprof = ctx.profile(reset=True)
    sweep_ms = sum(aprof.get(kk, {}).get("ms", 0.0) for kk in ("multidot", "multiaxpy"))
    sweep_bytes = k_adf * (k_adf + 1) * ctx.n * 16
    adf_sweeps = {"bytes_per_solve": sweep_bytes, "ms": round(sweep_ms, 3), "form": "delayed CGS2, two sweeps per step",
                  "GB_s": round(sweep_bytes / (sweep_ms * 1e6), 1) if sweep_ms else None,
                  "frac_hbm": round(sweep_bytes / (sweep_ms * 1e6) / hbm_peak, 3) if sweep_ms else None,
                  "classical_cgs2_bytes_equivalent_GB_s": round(2 * sweep_bytes / (sweep_ms * 1e6), 1) if sweep_ms else None,
                  "inner_sign_ms": round(aprof.get("inner_sign", {}).get("ms", 0.0), 3),
                  "stencil_ms": round(aprof.get("dslash", {}).get("ms", 0.0), 3)}
    # restarted Arnoldi: cycles of RS_M steps (a basis of RS_M + 1 double-float vectors instead of
    # k_adf + 1), the fewest cycles within 1e-8 of the FP64 k = 1000 solve and of the oracle
    ref1 = ctx.sign_krylov(ovl.LANCZOS2, K_REF, MU, KAPPA, b1)[0].clone()
    n1 = torch.linalg.vector_norm(ref1).item()
    rs_cyc, rs_err = None, None
    for cyc in range(2, RS_MAX_CYCLES + 1):
        y = ctx.sign_arnoldi_restarted(RS_M, cyc, MU, KAPPA, b1)[0]
        rs_err = torch.linalg.vector_norm(y - ref1).item() / n1
        rs_eo = None
        if oref is not None and rs_err <= 1e-8:
            d = oracle_error(y, oref)
            rs_eo = max(d["sampled_rel"], d["proj_rel"])
        print(f"[bench] calibrate arnoldi_restarted m={RS_M} cycles={cyc} err={rs_err:.3e} err_oracle={rs_eo}",
              file=sys.stderr, flush=True)
        if rs_err <= 1e-8 and (rs_eo is None or rs_eo <= 1e-8):
            rs_cyc = cyc
            break
    rs = {"m": RS_M, "cycles": rs_cyc, "rel_err_vs_k1000_fp64": rs_err,
          "basis_vectors": RS_M + 1, "basis_vectors_unrestarted": k_adf + 1}
    if rs_cyc is not None:
        t_rs = time_solves(torch, ctx, lambda b: ctx.sign_arnoldi_restarted(RS_M, rs_cyc, MU, KAPPA, b, out1,
                                                                            flags=ovl.OVERLAP), bsingle, 2, nctx, flush)
        rs.update(ms=statistics.mean(t_rs), solves_per_s=1e3 / statistics.mean(t_rs))
        if oref is not None:
            y = ctx.sign_arnoldi_restarted(RS_M, rs_cyc, MU, KAPPA, b1)[0]
            rs["vs_oracle_source_seed_2001"] = oracle_error(y, oref)
    # eigenvalues of D_ov nearest 0 (thick-restart Arnoldi, D_ov applied by mixed sign solves at the
    # calibrated k): wall time of the call (it synchronises once per restart), sign solves, residuals
    # (the residual each eigenpair has with D_ov applied by one FP64 solve at k = 1000 is reported
    # beside the solver's own check, which applies D_ov in mixed precision)
    ov = None
    try:
        vecs = torch.empty((OV_NEV, ctx.n), dtype=torch.complex128, device="cuda")
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        lam_ov, oinfo = ctx.overlap_eigs(ovl.LANCZOS2, k_s, MU, KAPPA, OV_NEV, flags=ovl.MIXED, tol=1e-7,
                                         maxit=40, vecs=vecs)
        sec = time.perf_counter() - t0
        r64 = 0.0
        for i in range(OV_NEV):
            dx = ctx.sign_krylov(ovl.LANCZOS2, K_REF, MU, KAPPA, vecs[i], flags=ovl.OVERLAP)[0]
            r64 = max(r64, (torch.linalg.vector_norm(dx - complex(lam_ov[i]) * vecs[i]) /
                            torch.linalg.vector_norm(vecs[i])).item())
        ov = {"nev": OV_NEV, "k": k_s, "flags": "mixed two-pass sign solves", "tol": 1e-7, "seconds": round(sec, 3),
              "nearest": [[round(z.real, 10), round(z.imag, 10)] for z in lam_ov[:3]],
              "ms_per_sign_solve": round(1e3 * sec / max(oinfo["sign_solves"], 1), 3), **oinfo,
              "max_residual_fp64_k1000_check": r64}
        del vecs
    except Exception as exc:  # report, keep the rest of the line
        ov = {"error": repr(exc)[:200]}
    res = {
        "workload": WORKLOAD8, "deflation_setup": eig,
        "batch_mixed": {"solves_per_s": NRHS * 1e3 / statistics.mean(t_b), "ms_per_batch": statistics.mean(t_b),
                        "k": k_mix, "max_rel_err_vs_k1000_fp64": err_mix,
                        "method": "batched two-sided Lanczos, FP32 pass 1 (persistent), double-float pass 2"},
        "batch_fp64": {"solves_per_s": NRHS * 1e3 / statistics.mean(t_b64), "ms_per_batch": statistics.mean(t_b64),
                       "k": k_64, "max_rel_err_vs_k1000_fp64": err_64},
        "single_mixed": {"solves_per_s": 1e3 / statistics.mean(t_s), "ms": statistics.mean(t_s), "k": k_s,
                         "rel_err_vs_k1000_fp64": err_s, "kernels": "persistent passes (FP32 pass 1, FP64 pass 2)",
                         "profile_ms_by_kernel_class": single_profile, "with_reprojection": reproj},
        "single_fp64": {"solves_per_s": 1e3 / statistics.mean(t_s64), "ms": statistics.mean(t_s64), "k": k_s64,
                        "rel_err_vs_k1000_fp64": err_s64},
        "arnoldi_fp64": {"solves_per_s": 1e3 / statistics.mean(t_arn), "ms": statistics.mean(t_arn), "k": k_arn,
                         "rel_err_vs_k1000_fp64": err_arn,
                         "k_ratio_2sl_over_arnoldi": (k_s64 / k_arn) if k_arn else None},
        "arnoldi_doublefloat": {"solves_per_s": 1e3 / statistics.mean(t_adf), "ms": statistics.mean(t_adf),
                                "k": k_adf, "rel_err_vs_k1000_fp64": err_adf, "gram_schmidt_sweeps": adf_sweeps},
        "arnoldi_restarted": rs,
        "overlap_eigenvalues": ov,
        "vs_oracle_source_seed_2001": vs_oracle,
    }
    bt.close()
    ctx.close()
    torch.cuda.empty_cache()
    return res, U


def config3_extra(torch, ovl, flush, steps):
    """16^3 x 8, mu = 0.3, 30 deflated eigenpairs: single-source mixed precision at the smallest k
    on a grid (step 10, at most 800) within 1e-8 of the FP64 k = 1200 solve, against FP64 at its own
    calibrated k; the error of each stated against the FP64 reference."""
    from paper_0810_4228_gb300 import synth
    ctx = ovl.Context(C3_DIMS)
    ctx.set_gauge(torch.from_numpy(synth.gauge_field(C3_DIMS, EPS, C3_SEED_U)).cuda())
    t0 = time.perf_counter()
    eig = ctx.deflation_eigs(C3_MU, KAPPA, C3_M)
    eig["seconds"] = round(time.perf_counter() - t0, 2)
    b = torch.from_numpy(synth.gaussian_source(C3_DIMS, C3_SEED_B)).cuda()
    ref = ctx.sign_krylov(ovl.LANCZOS2, 1200, C3_MU, KAPPA, b)[0].clone()
    nrm = torch.linalg.vector_norm(ref).item()
    out = {"dims": list(C3_DIMS), "mu": C3_MU, "m": C3_M, "deflation_setup": eig,
           "reference": "FP64 two-sided Lanczos, k = 1200"}
    for name, fl in (("mixed", ovl.MIXED), ("fp64", 0)):
        chosen, err = 800, None
        for k in range(400, 801, 10):
            y = ctx.sign_krylov(ovl.LANCZOS2, k, C3_MU, KAPPA, b, flags=fl)[0]
            err = torch.linalg.vector_norm(y - ref).item() / nrm
            if err <= 1e-8:
                chosen = k
                break
        y1 = torch.empty_like(b)
        t = time_solves(torch, ctx, lambda bb: ctx.sign_krylov(ovl.LANCZOS2, chosen, C3_MU, KAPPA, bb, y1,
                                                               flags=fl | ovl.OVERLAP), [b], 2, max(3, steps), flush)
        out[name] = {"k": chosen, "rel_err_vs_fp64_k1200": err, "ms": statistics.mean(t),
                     "solves_per_s": 1e3 / statistics.mean(t)}
    ctx.close()
    torch.cuda.empty_cache()
    return out


def run_ours(args, world, rank, local):
    import torch
    from paper_0810_4228_gb300 import ovl, synth

    torch.cuda.set_device(local)
    if args.dw_only:
        ovl.load()
        dims = tuple(int(v) for v in args.dw_dims.split(",")) if args.dw_dims else DW_DIMS
        ddims, dV, dres = dw_bandwidth(torch, ovl, reps=args.steps, dims=dims)
        print(json.dumps({"dw_only": True, "dims": list(ddims), "sites": dV,
                          **{nm: {"ms": r["ms"], "GB_s": r["GB_s"]} for nm, r in dres.items()}}))
        return
    if args.arnoldi_only:
        # single-source Arnoldi with the double-float basis on the 8^4 workload (for profiler
        # captures of its Gram-Schmidt sweeps): `--steps` solves at `--k` (default 450), `--m` deflated
        ovl.load()
        ctx = ovl.Context(DIMS)
        ctx.set_gauge(torch.from_numpy(synth.gauge_field(DIMS, EPS, SEED_U)).cuda())
        if args.m > 0:
            ctx.deflation_eigs(MU, KAPPA, args.m)
        b = torch.from_numpy(synth.gaussian_source(DIMS, SEED_B)).cuda()
        y = torch.empty_like(b)
        ka = args.k or 450
        flush = torch.empty(512 << 20, dtype=torch.uint8, device="cuda")
        t = time_solves(torch, ctx, lambda bb: ctx.sign_krylov(ovl.ARNOLDI, ka, MU, KAPPA, bb, y,
                                                               flags=ovl.MIXED | ovl.OVERLAP), [b], args.warmup,
                        args.steps, flush)
        print(json.dumps({"arnoldi_only": True, "k": ka, "m": args.m, "ms": statistics.mean(t)}))
        return
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    ovl.load()
    hbm_peak, peak_kind = peaks()
    flush = torch.empty(512 << 20, dtype=torch.uint8, device="cuda")
    orefs = load_oracle_refs()
    orefs_head = {n: r for n, r in orefs.items() if n.startswith("batch")} if rank == 0 else {}

    # ---- headline: deflation set-up (untimed), the batch of 48 sequences
    ctxs, srcs, setup = headline_setup(torch, ovl, args.head_m)
    if rank > 0:  # replicas: each rank its own point sources (site = rank)
        srcs = [torch.from_numpy(synth.point_sources(d, site=rank % (d[0] * d[1] * d[2] * d[3]))).cuda()
                for d in HEAD_DIMS]
    print(f"[bench] headline deflation {setup}", file=sys.stderr, flush=True)
    bt = ovl.Batch(ctxs, [NRHS] * len(ctxs))
    nseq = NRHS * len(ctxs)
    sites = [d[0] * d[1] * d[2] * d[3] for d in HEAD_DIMS]
    seq_sites = NRHS * sum(sites)
    fl_mix, fl_64 = ovl.MIXED | ovl.OVERLAP, ovl.OVERLAP

    if args.solves_only:
        if not args.k:
            raise SystemExit("--solves-only needs --k")
        outs = [s.clone() for s in srcs]
        t = time_solves(torch, None, lambda _: bt.solve(args.k, HEAD_MU, KAPPA, srcs, outs, flags=fl_mix), [0],
                        args.warmup, args.steps, flush)
        if args.profile_one:
            # one more solve between cudaProfilerStart/Stop: `ncu --profile-from-start off` captures
            # exactly the launches of one solve (no effect without a profiler)
            torch.cuda.synchronize()
            torch.cuda.cudart().cudaProfilerStart()
            bt.solve(args.k, HEAD_MU, KAPPA, srcs, outs, flags=fl_mix)
            torch.cuda.synchronize()
            torch.cuda.cudart().cudaProfilerStop()
        print(json.dumps({"solves_only": True, "k": args.k, "ms_per_step": statistics.mean(t),
                          "solves_per_s": nseq * 1e3 / statistics.mean(t)}))
        return

    # ---- accuracy calibration (untimed)
    refs64 = None
    if args.k:
        k_mix, err64_mix, erro_mix, ref_vs_oracle = args.k, None, None, None
    else:
        k_mix, err64_mix, erro_mix, ref_vs_oracle, refs64 = calibrate_headline(
            torch, ovl, bt, ctxs, srcs, orefs_head, ovl.MIXED, HEAD_K_GRID)
    print(f"[bench] headline k={k_mix} err_fp64={err64_mix} err_oracle={erro_mix}", file=sys.stderr, flush=True)

    # ---- per-phase profile of the batched solve (CUDA events around each phase, eager launches)
    outs = [torch.empty_like(s) for s in srcs]
    nprof = 3
    bt.profile(reset=True)
    for _ in range(nprof):
        _, pinfo, _ = bt.solve(k_mix, HEAD_MU, KAPPA, srcs, outs, flags=fl_mix | ovl.PROFILE)
    prof, _ = bt.profile(reset=True)
    prof = {kk: v / nprof for kk, v in prof.items()}
    tuned = bt.tuning()
    kused = max(i["k_used"] for i in pinfo)
    print(f"[bench] batch profile {prof}", file=sys.stderr, flush=True)

    # ---- timed region: the mixed batched solve (headline), device-resident inputs
    clocks = Clocks(local)
    if world > 1:
        torch.distributed.barrier()
    torch.cuda.synchronize()
    clocks.start()
    t_mix = time_solves(torch, None, lambda _: bt.solve(k_mix, HEAD_MU, KAPPA, srcs, outs, flags=fl_mix), [0],
                        args.warmup, args.steps, flush)
    torch.cuda.synchronize()
    clk = clocks.stop()
    tot = max_over_ranks(sum(t_mix), world, "cuda")
    if world > 1:
        torch.distributed.barrier()
    value = whole_job_rate(tot, world, nseq, args.steps)
    print(f"[bench] headline mixed solves/s {value:.2f}, ms/step {statistics.mean(t_mix):.3f}, steps "
          f"{[round(t, 3) for t in t_mix]}", file=sys.stderr, flush=True)

    # ---- end to end through the C ABI with host buffers (copies inside the timed region)
    hsrc = [s.cpu().pin_memory() for s in srcs]
    hout = [torch.empty_like(h).pin_memory() for h in hsrc]
    t_e2e = time_solves(torch, None, lambda _: bt.solve(k_mix, HEAD_MU, KAPPA, hsrc, hout, flags=fl_mix), [0],
                        args.warmup, args.steps, flush)
    e2e_val = whole_job_rate(max_over_ranks(sum(t_e2e), world, "cuda"), world, nseq, args.steps)
    nbytes = sum(s.numel() * s.element_size() for s in srcs)

    # ---- the same batch in FP64 at equal accuracy (smallest k on the grid from k_mix - 100 up)
    fp64 = None
    try:
        if refs64 is not None:
            k64, e64 = HEAD_K_GRID[-1], None
            for k in [kk for kk in HEAD_K_GRID if kk >= k_mix - 100]:
                o64, _, _ = bt.solve(k, HEAD_MU, KAPPA, srcs, flags=0)
                e64, eo64 = headline_errors(torch, o64, refs64, orefs_head)
                if e64 <= 1e-8 and (eo64 is None or eo64 <= 1e-8):
                    k64 = k
                    break
            del o64
        else:
            k64, e64 = k_mix, None
        t64 = time_solves(torch, None, lambda _: bt.solve(k64, HEAD_MU, KAPPA, srcs, outs, flags=fl_64), [0], 1,
                          max(2, min(args.steps, 3)), flush)
        fp64 = {"k": k64, "max_rel_err_vs_k1500_fp64": e64, "ms_per_batch": statistics.mean(t64),
                "solves_per_s": nseq * 1e3 / statistics.mean(t64),
                "method": "batched two-sided Lanczos in FP64, two passes (the stored basis would exceed 32 GiB)"}
    except Exception as exc:  # report, keep the headline measurement
        fp64 = {"error": repr(exc)[:200]}
    del refs64
    torch.cuda.empty_cache()

    # ---- roofline of the dominant phase (algorithmic bytes of the method, Sec. 4-5)
    steps2 = max(kused - 1, 1)
    roof_all = {
        "pass1_batched_fp32": {"bound": "hbm", "achieved": PASS1_BYTES_SITE * seq_sites * kused / prof["pass1"] / 1e6,
                               "peak": hbm_peak, "unit": "GB/s",
                               "algorithmic": f"{PASS1_BYTES_SITE} B/site/step x {seq_sites} site-sequences x {kused} steps",
                               "ms_per_launch_sequence": prof["pass1"],
                               "kernels": "k_b_pair + k_b_lstep per step"},
        "pass2_batched_doublefloat": {
            "bound": "hbm", "achieved": PASS2_BYTES_SITE * seq_sites * steps2 / prof["pass2_or_combine"] / 1e6,
            "peak": hbm_peak, "unit": "GB/s",
            "algorithmic": f"{PASS2_BYTES_SITE} B/site/step x {seq_sites} site-sequences x {steps2} steps",
            "ms_per_launch_sequence": prof["pass2_or_combine"], "kernels": "k_b_regen_df per step",
            "alu_view": {
                "fp32_ops_achieved_T": REGEN_DFX_OPS_SITE * seq_sites * steps2 / prof["pass2_or_combine"] / 1e9,
                "fp32_issue_peak_T": FP32_OPS_PEAK_T,
                "note": f"{REGEN_DFX_OPS_SITE} FP32 operations/site/step of the double-float arithmetic",
                "fp64_equivalent_tflops": REGEN_FLOP_SITE * seq_sites * steps2 / prof["pass2_or_combine"] / 1e9,
                "fp64_roof_tflops": FP64_PEAK_TFLOPS}},
    }
    for r_ in roof_all.values():
        r_["frac"] = r_["achieved"] / r_["peak"]
        if "alu_view" in r_:
            av = r_["alu_view"]
            av["frac_fp32_issue"] = av["fp32_ops_achieved_T"] / av["fp32_issue_peak_T"]
    dname = "pass2_batched_doublefloat" if prof["pass2_or_combine"] >= prof["pass1"] else "pass1_batched_fp32"
    roof = dict(roof_all[dname])
    roof.update({"kernel": dname, "traffic": HEAD_TRAFFIC.get(dname),
                 "peak_kind": f"{peak_kind} hbm_gbs (MEASURED_PEAKS.json)"})

    # ---- extras (rank 0)
    extras = {}
    if rank == 0 and not args.no_extras:
        for key, fn in (("config_16x3x8_m30", lambda: config3_extra(torch, ovl, flush, args.steps)),
                        ("gauss8", lambda: gauss8_extras(torch, ovl, args, flush, orefs, hbm_peak, rank))):
            try:
                extras[key] = fn()
            except Exception as exc:  # report, keep the headline measurement
                extras[key] = {"error": repr(exc)[:200]}
        U8 = None
        if isinstance(extras.get("gauss8"), tuple):
            extras["gauss8"], U8 = extras["gauss8"]
        if not args.no_grad and U8 is not None:
            try:
                extras["autograd"] = autograd_timing(
                    torch, ovl, U8, torch.from_numpy(synth.gaussian_source(DIMS, SEED_B)).cuda(), flush)
            except Exception as exc:  # report, keep the headline measurement
                extras["autograd"] = {"error": repr(exc)[:200]}
    dw = None
    single_large = {}
    if rank == 0 and not args.no_dw:
        try:
            ddims, dV, dres = dw_bandwidth(torch, ovl, single_source=single_large)
        except Exception as exc:  # report, keep the solve measurement
            dres, ddims, dV = {}, DW_DIMS, 0
            dw = {"error": repr(exc)[:200]}
        dw = dw or {"dims": list(ddims), "sites": dV}
        for nm, r in dres.items():
            dw[nm] = {"ms": round(r["ms"], 4), "GB_s": round(r["GB_s"], 1), "frac_hbm": round(r["GB_s"] / hbm_peak, 3),
                      "GFLOP_s": round(r["GFLOP_s"], 1)}
            if nm == "f64":
                dw[nm]["frac_fp64_roof"] = round(r["GFLOP_s"] / (FP64_PEAK_TFLOPS * 1e3), 3)
            if tuple(ddims) == DW_DIMS and nm in DW_TRAFFIC:
                dw[nm]["traffic"] = DW_TRAFFIC[nm]
                dw[nm]["traffic_over_algorithmic"] = round(DW_TRAFFIC[nm] / (DW_BYTES[nm] * dV), 3)
        dw["hbm_peak_gbs"] = hbm_peak
        if single_large:
            dw["single_source_mixed"] = single_large

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu:
        try:
            cpu = oracle_batch_sample(k_mix, budget_s=15.0)
        except Exception as exc:  # report, keep the headline measurement
            cpu = {"error": repr(exc)[:200]}

    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": "solves/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": statistics.mean(t_mix),
            "ms_per_step_median": statistics.median(t_mix), "ms_per_step_min": min(t_mix), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f32+f64", "data": "synthetic",
            "config": {"workload": HEAD_WORKLOAD, "dims": [list(d) for d in HEAD_DIMS], "mu": HEAD_MU,
                       "kappa": KAPPA, "eps": EPS, "rhs_per_lattice": NRHS, "sequences_per_step": nseq,
                       "autotuned_shapes": {"pass1_sites_per_block": tuned[0], "regen_blocks_per_sm": tuned[1],
                                            "regen_sequences_per_block": tuned[2]} if tuned else None,
                       "method": ("batched two-sided Lanczos, two-pass mixed: FP32 pass 1 (12-real links), "
                                  "double-float pass 2 (about 48 significant bits), FP64 coefficients"),
                       "k": k_mix, "m_deflated": args.head_m, "deflation_setup": setup,
                       "max_rel_err_vs_k1500_fp64": err64_mix,
                       "max_rel_err_vs_oracle": erro_mix,
                       "oracle_sources": sorted(orefs_head),
                       "k1500_fp64_reference_vs_oracle": ref_vs_oracle,
                       "l2": "flushed (512 MiB write) before every timed step", "parallelism": f"replicas x{world}"},
            "roofline": roof,
            "roofline_phases": roof_all,
            "cpu_baseline": cpu,
            "e2e": {"value": e2e_val, "unit": "solves/s", "h2d_bytes_per_step": nbytes,
                    "d2h_bytes_per_step": nbytes},
            "gpu_launches": headline_launches(k_mix, args.head_m, fused_start=True) * args.steps,
            "clocks": clk,
            "profile_ms_per_batch": {kk: round(v, 4) for kk, v in prof.items()},
            "fp64_batched": fp64,
            **extras,
            "dw": dw,
        }
        print(json.dumps(line))
    bt.close()
    for c in ctxs:
        c.close()
    if world > 1:
        torch.distributed.destroy_process_group()


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--k", type=int, default=0, help="fix the Krylov size (skip the accuracy calibration)")
    ap.add_argument("--m", type=int, default=M_DEFL, help="deflated eigenpairs of the 8^4 extras (0: none)")
    ap.add_argument("--head-m", type=int, default=HEAD_M,
                    help="deflated eigenpairs per lattice of the headline batch (profiler runs may pass 0)")
    ap.add_argument("--no-dw", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--no-extras", action="store_true", help="only the headline batch (and the stencil bandwidth)")
    ap.add_argument("--no-grad", action="store_true", help="skip the gradient timings")
    ap.add_argument("--dw-only", action="store_true", help="only the stencil bandwidth measurement (--steps repetitions)")
    ap.add_argument("--dw-dims", default="", help="lattice of the stencil bandwidth measurement, e.g. 32,32,32,32")
    ap.add_argument("--profile-one", action="store_true",
                    help="with --solves-only: one extra solve inside cudaProfilerStart/Stop (for ncu)")
    ap.add_argument("--arnoldi-only", action="store_true",
                    help="only single-source double-float Arnoldi solves on 8^4 (for profiler captures)")
    ap.add_argument("--solves-only", action="store_true",
                    help="only the timed headline solves (for profiler captures): needs --k, skips calibration, "
                         "profile, e2e, extras, the bandwidth lattice and the CPU baseline")
    args = ap.parse_args()
    world, rank, local = dist_setup()
    if args.impl == "reference":
        run_reference(args, world, rank)
        return
    run_ours(args, world, rank, local)


if __name__ == "__main__":
    main()
