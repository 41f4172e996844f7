#!/usr/bin/env python
"""Benchmark of the DPR1 eigensolver on GB300: eigenpairs/s for the n = 16384 hard-spectrum
forward solve (eigenvalues and the full eigenvector matrix, binary64).

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

For N > 1 run under torch.distributed.run: every rank solves its own independent problem
of the same workload (weak scaling, no collective on the data path); the reported value
is all eigenpairs of all ranks divided by the slowest rank's time.

One JSON line is printed by rank 0.  Timing: W untimed warm-up steps, then K steps, each
a full dpr1_eig call timed with CUDA events on the launching stream, L2 flushed (256 MiB
write) before every step outside the timed events; nvidia-smi clocks are sampled during
the timed region.  The line carries the roofline of the solve kernel (algorithmic binary64
operations over its event-timed duration, against the nominal peak; DRAM traffic from the
committed ncu record while the kernel sources are unchanged), that of the eigenvector phase
(the n^2 write of V against the measured copy rate, and its binary64 work), the CPU oracle on a bounded
sample (all host cores, and one thread on a smaller sample), the end-to-end rate through the binding from pinned host buffers (double-buffered
outputs), and extra measurements (--extras; --only runs one alone at size --n):
  small          the n = 512 forward, direct calls and a CUDA-graph replay
  fwd_bwd        forward and adjoint at n = 4096
  fwd_bwd_large  forward and adjoint with recompute at n = 32768 (W drawn on the device)
  batched        4096 uneven problems in one graph replay against a per-problem loop
  accel          the same workload with the accelerated bracketed solve
  hermitian      the complex Hermitian problem (hard spectrum with random phases)
  tridiag        divide and conquer for a random tridiagonal matrix, n = 4096
  arrow          the arrowhead eigenproblem, n = 16384 poles
``--impl reference`` times the CPU oracle (Algorithm 1 in binary64 on the host cores) on
bounded samples of the same workload.
"""
import argparse
import hashlib
import json
import math
import os
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

METRIC = "DPR1 eigenpairs/s at n=16384 FP64, % roofline; fwd+bwd and batched vs plain"
N_DEFAULT = 16384
SEED = 1
RHO = 1e3
# binary64 peak derived from the nominal GB300 figure of 1.25 TFLOP/s: 0.625e12 fma/s, i.e.
# 2 binary64 instructions per clock per SM on 152 SMs at the 2070 MHz maximum clock
NOMINAL_FP64_OPS = 2 * 152 * 2070e6
# algorithmic binary64 operations per secular term (sub, fma, mul, div, add; fma and div = 1 op)
OPS_PER_TERM = 5          # a secular term: sub, fma, mul, div, add
ACCEL_OPS_PER_TERM = 8    # the same with its slope (mul, mul, fma)
# a double-double term zeta_j^2 / (d_j - d_i) of the corner b: TwoSum of the difference (6),
# TwoProd of the square (2), quotient and its first-order correction (5), compensated
# accumulation (7)
DD_OPS_PER_TERM = 20
# binary32 operations per term of the screens (screen_sum: the term's fma, the Newton step of the
# reciprocal, the quotient, w, the compensated sum and the bound; screen_df_sum: the double-float
# term, its division and three TwoSum levels with the running bound), and the weight of a binary32
# operation against a binary64 one: 128 binary32 lanes against 2 binary64 lanes per SM and clock
B32_OPS_PER_TERM = 14
DF_OPS_PER_TERM = 50
FP32_PER_FP64 = 64
# the binary64 pass over the corner's terms that decides whether b needs double-double
# (kappa_nu of Eq. (knu2)): sub, div, mul, add
B64_OPS_PER_TERM = 4
# the binary32 pass of the shift test (shift_test_f32): per term 16 binary32 operations (difference,
# reciprocal and its Newton step, quotient, w, the bound's two fma, the magnitude sum, TwoSum and the
# low-part sum); the poles' difference is integer work, so no binary64 operation
SHIFT32_B64_OPS_PER_TERM = 0
SHIFT32_OPS_PER_TERM = 16
# an eigenvector component (Eq. (eigenvecAi)): 2 sub, 1 div, 1 mul, 1 fma (sum of squares), 1 mul
# (rescale); the solve kernel's lane groups write rows once its queue is empty
VEC_OPS_PER_ELEMENT = 6


def shift_test_ops(n, stats, screen=True):
    """Binary64 and binary32 operations of the shift tests of one launch (Algorithm 1, the
    choice of the pole): the eigenvalues k >= 1 each take the binary32 pass (with the screen
    on) and, where its bound does not settle the sign, the 5-op binary64 pass."""
    tests = n - 1
    s32 = stats.get("shift_binary32", 0) if screen else 0
    ops64 = (n - 1) * (OPS_PER_TERM * (tests - s32) + (SHIFT32_B64_OPS_PER_TERM * tests if screen else 0))
    ops32 = (n - 1) * SHIFT32_OPS_PER_TERM * tests if screen else 0
    return ops64, ops32
# kernels one dpr1_eig call launches: k_norm, k_scan, k_deflate, k_solve, k_classify, k_fix, k_zero_detect,
# k_zero_solve, k_defl_positions, k_vectors, k_defl_rows, k_trivial
LAUNCHES_PER_CALL = 12


def workload_config(n):
    return {"workload": "DPR1 forward, hard spectrum: half the poles graded 10^(-12 j/n), half U(-1,1), "
                        "gaps >= 1e-14; |z| log-uniform [1e-10, 1], random sign; rho = 1e3; eigenvalues "
                        "and full V",
            "n": n, "rho": RHO, "seed": SEED, "dtype": "binary64",
            "l2": "flushed before every timed step (256 MiB write); V (8 n^2 B) exceeds L2"}


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--n", type=int, default=N_DEFAULT)
    ap.add_argument("--e2e-steps", type=int, default=20,
                    help="end-to-end steps; the last step's copy of V back to the host is not overlapped")
    ap.add_argument("--cpu-sample", type=int, default=8192)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-extras", action="store_true",
                    help="skip the batched-vs-loop and forward+backward measurements")
    ap.add_argument("--extras", default="small,fwd_bwd,fwd_bwd_large,batched,accel,hermitian,tridiag,arrow",
                    help="comma list of extra measurements: small, fwd_bwd, fwd_bwd_large, batched, accel, "
                         "hermitian, tridiag, arrow")
    ap.add_argument("--only", choices=["tridiag", "hermitian", "fwd_bwd", "arrow"], default=None,
                    help="run one extra measurement alone at size --n (a small case for profiling) and print it")
    ap.add_argument("--zero-finder", type=int, choices=[0, 1], default=0,
                    help="0: bisection (the method as stated, default); 1: the accelerated bracketed solve")
    return ap.parse_args()


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


# ------------------------------------------------------------------ clocks
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "--query-gpu=" + self.FIELDS, "--format=csv,noheader,nounits",
                                          "-lms", "200"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except (OSError, ValueError):
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            out, _ = self.proc.communicate(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
            out, _ = self.proc.communicate()
        sm, smax, reasons, power = [], [], set(), []
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in out.splitlines():
            p = [x.strip() for x in line.split(",")]
            if len(p) < 9:
                continue
            try:
                if int(p[0]) != self.gpu:
                    continue
                sm.append(float(p[1]))
                smax.append(float(p[2]))
                power.append(float(p[3]))
            except ValueError:
                continue
            for nm, v in zip(names, p[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(smax), "reasons": sorted(reasons),
                "samples": len(sm), "power_w_max": max(power) if power else None}


# ------------------------------------------------------------------ reference (CPU oracle) arm
def cpu_oracle_rate(d, z, rho, nsample, seed=7, threads=None):
    import oracle
    threads = threads or os.cpu_count() or 1
    rng = np.random.default_rng(seed)
    ks = np.sort(rng.choice(d.size, size=min(nsample, d.size), replace=False))
    t0 = time.perf_counter()
    oracle.eig_all(d, z, rho, ks=ks, threads=threads)
    dt = time.perf_counter() - t0
    return ks.size / dt, threads, ks.size, dt


def run_reference(args):
    ws, rank, _ = dist_env()
    if rank != 0:
        return 0
    from paper_1405_7537_gb300 import workloads as W
    d, z, rho = W.hard(args.n, SEED)
    # a sample large enough that thread start-up on the host cores is negligible (about a third of
    # a second of oracle work per step on 16 cores)
    per_step = 2048
    for _ in range(args.warmup):
        cpu_oracle_rate(d, z, rho, per_step, seed=99)
    times = []
    threads = os.cpu_count() or 1
    for s in range(args.steps):
        _, threads, m, dt = cpu_oracle_rate(d, z, rho, per_step, seed=1000 + s)
        times.append(dt)
    total = sum(times)
    value = per_step * args.steps / total
    line = {"metric": METRIC, "value": value, "unit": "eigenpairs/s", "n_gpus": args.gpus, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": 1e3 * total / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": dict(workload_config(args.n), zero_finder="bisection"), "impl": "reference",
            "cpu_baseline": {"value": value, "unit": "eigenpairs/s", "cores": threads, "kind": "oracle",
                             "sample": "%d random eigenpairs of the n=%d workload per step, all host cores"
                                       % (per_step, args.n)},
            "e2e": {"value": value, "unit": "eigenpairs/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


# ------------------------------------------------------------------ multi-rank aggregation
def aggregate(total_ms, units_per_rank, steps, world, dist=None, device="cpu"):
    """Whole-job rate over `world` ranks that each processed `units_per_rank` units per step:
    the slowest rank's time (max over ranks) divides all ranks' units.  Returns
    (value, max_ms)."""
    if world > 1:
        import torch
        t = torch.tensor([float(total_ms)], dtype=torch.float64, device=device)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        total_ms = t.item()
    return world * units_per_rank * steps / (total_ms * 1e-3), total_ms


# ------------------------------------------------------------------ extras
def _events():
    import torch
    return torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)


def bench_batched(B, dev, steps):
    """4096 uneven problems: one graph-captured dpr1_eig_batched vs a loop of dpr1_eig calls."""
    import torch
    from paper_1405_7537_gb300 import tune
    from paper_1405_7537_gb300 import workloads as W
    offs, d, z, rho = W.batch()
    sizes = np.diff(offs)
    bt = B.Batch(sizes, device=dev)
    dt = torch.tensor(d, device=dev)
    zt = torch.tensor(z, device=dev)
    rt = torch.tensor(rho, device=dev)
    shape = tune.tune(sizes, device=dev)
    opts = B.default_options(lanes=shape[0], warps_per_block=shape[1], blocks_per_sm=shape[2])
    side = torch.cuda.Stream(device=dev)
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        bt.solve(dt, zt, rt, options=opts)
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    st = B.stream_status(bt.ws)
    if st != 0:
        raise B.DPR1Error(st, "batched warm-up")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        bt.solve(dt, zt, rt, options=opts)
    g.replay()
    torch.cuda.synchronize()
    ms = []
    for _ in range(max(1, steps)):
        e0, e1 = _events()
        e0.record()
        g.replay()
        e1.record()
        e1.synchronize()
        ms.append(e0.elapsed_time(e1))
    batched_ms = statistics.mean(ms)
    # the same graph-captured launch with the accelerated bracketed solve
    shape_a = tune.tune(sizes, device=dev, zero_finder=B.ACCELERATED)
    opts_a = B.default_options(lanes=shape_a[0], warps_per_block=shape_a[1], blocks_per_sm=shape_a[2],
                               zero_finder=B.ACCELERATED)
    with torch.cuda.stream(side):
        bt.solve(dt, zt, rt, options=opts_a)
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    st = B.stream_status(bt.ws)
    if st != 0:
        raise B.DPR1Error(st, "batched accelerated warm-up")
    ga = torch.cuda.CUDAGraph()
    with torch.cuda.graph(ga):
        bt.solve(dt, zt, rt, options=opts_a)
    ga.replay()
    torch.cuda.synchronize()
    ms_a = []
    for _ in range(max(1, steps)):
        e0, e1 = _events()
        e0.record()
        ga.replay()
        e1.record()
        e1.synchronize()
        ms_a.append(e0.elapsed_time(e1))
    accel_ms = statistics.mean(ms_a)
    # the same problems, one dpr1_eig call each (default launch shape, shared workspace)
    ws = B.workspace(int(sizes.max()), dev)
    lam, Vt = bt.lam, bt.Vt
    outs = []
    for p in range(bt.P):
        a, b = int(offs[p]), int(offs[p + 1])
        n = b - a
        va = int(bt.voffs_host[p])
        outs.append((dt[a:b], zt[a:b], float(rho[p]),
                     dict(lam=lam[a:b], Vt=Vt[va:va + n * n].view(n, n), sigma=bt.sigma[a:b], mu=bt.mu[a:b],
                          xnorm=bt.xnorm[a:b])))
    for dp, zp, rp, out in outs[:64]:
        B.eig(dp, zp, rp, ws=ws, out=out, check=False)
    torch.cuda.synchronize()
    e0, e1 = _events()
    e0.record()
    for dp, zp, rp, out in outs:
        B.eig(dp, zp, rp, ws=ws, out=out, check=False)
    e1.record()
    e1.synchronize()
    loop_ms = e0.elapsed_time(e1)
    total = int(offs[-1])
    return {"workload": "4096 problems, n_k = round(exp(U(ln 16, ln 2048))), d, z ~ U(-1,1), rho_k ~ U(0.1, 10), "
                        "seed 3; eigenvalues and all V blocks",
            "eigenpairs": total, "v_bytes": int(bt.voffs_host[-1]) * 8,
            "batched_ms": batched_ms, "value": total / (batched_ms * 1e-3),
            "loop_ms": loop_ms, "loop_value": total / (loop_ms * 1e-3),
            "speedup_vs_loop": loop_ms / batched_ms, "unit": "eigenpairs/s",
            "accelerated_ms": accel_ms, "accelerated_value": total / (accel_ms * 1e-3),
            "launch": "one CUDA-graph replay of dpr1_eig_batched vs 4096 dpr1_eig calls from Python",
            "tuned_shape": {"lanes": shape[0], "warps_per_block": shape[1], "blocks_per_sm": shape[2]},
            "tuned_shape_accelerated": {"lanes": shape_a[0], "warps_per_block": shape_a[1], "blocks_per_sm": shape_a[2]}}


def bench_fwd_bwd(B, dev, n, seed, steps, with_w):
    """Forward (lambda and V) and backward (recomputing V) times for loss = w.lambda + sum W o V."""
    import torch
    from paper_1405_7537_gb300 import workloads as W
    if with_w:
        d, z, rho, w, Wm = W.diff(n, seed)
        gVt = torch.tensor(Wm.T.copy(), device=dev)        # dL/dVt = W^T for V[:, k] = v_k
        del Wm
    else:
        # n = 32768: W ~ N(0, 1) (8.6 GB) is drawn on the device from a seeded generator; the
        # backward reads it once like any dL/dVt
        d, z, rho, _ = W.large(n, seed, with_W=False)
        w = None
        gen = torch.Generator(device=dev)
        gen.manual_seed(seed)
        gVt = torch.randn((n, n), dtype=torch.float64, device=dev, generator=gen)
    dt = torch.tensor(np.array(d), device=dev)
    zt = torch.tensor(np.array(z), device=dev)
    wt = torch.tensor(w, device=dev) if w is not None else None
    ws = B.workspace(n, dev)
    bws = B.backward_workspace(n, dev)
    out = B.eig(dt, zt, rho, ws=ws)
    B.eig_backward(dt, zt, rho, out["sigma"], out["mu"], wt, gVt, ws=bws)
    torch.cuda.synchronize()
    fw, bw = [], []
    for _ in range(max(1, steps)):
        e0, e1 = _events()
        e2, e3 = _events()
        e0.record()
        B.eig(dt, zt, rho, ws=ws, out=out, check=False)
        e1.record()
        e2.record()
        B.eig_backward(dt, zt, rho, out["sigma"], out["mu"], wt, gVt, ws=bws, check=False)
        e3.record()
        e3.synchronize()
        fw.append(e0.elapsed_time(e1))
        bw.append(e2.elapsed_time(e3))
    f, b = statistics.mean(fw), statistics.mean(bw)
    del gVt
    return {"n": n, "seed": seed, "fwd_ms": f, "bwd_ms": b, "fwd_plus_bwd_over_fwd": (f + b) / f,
            "value": n / ((f + b) * 1e-3), "unit": "eigenpairs/s (forward + backward)", "steps": max(1, steps),
            "loss": ("w . lambda + " if with_w else "") + "sum W o V, W ~ N(0,1)"
                    + ("" if with_w else " (drawn on the device, torch generator seed %d)" % seed),
            "note": "the backward recomputes the eigenvector columns from (sigma, mu); V is not saved"}


def bench_small(B, dev, steps):
    """The n = 512 forward (d, z ~ U(-1, 1), rho = 1, seed 0; eigenvalues and V): back-to-back
    dpr1_eig calls, and the same call captured once in a CUDA graph and replayed.  At this size a
    call is a dozen short launches, so the graph shows what launch overhead costs."""
    import torch
    from paper_1405_7537_gb300 import workloads as W
    d, z, rho = W.uniform(512, 0)
    n = d.size
    dt = torch.tensor(d, device=dev)
    zt = torch.tensor(z, device=dev)
    ws = B.workspace(n, dev)
    out = B.eig(dt, zt, rho, ws=ws)
    torch.cuda.synchronize()
    reps = 200
    res = {"workload": "n=512, d, z ~ U(-1,1) (|z| > 1e-3), rho = 1, seed 0; eigenvalues and V", "n": n,
           "unit": "eigenpairs/s", "calls_per_step": reps}
    ms = []
    for _ in range(max(1, steps)):
        e0, e1 = _events()
        e0.record()
        for _ in range(reps):
            B.eig(dt, zt, rho, ws=ws, out=out, check=False)
        e1.record()
        e1.synchronize()
        ms.append(e0.elapsed_time(e1) / reps)
    t = statistics.mean(ms)
    res["direct"] = {"value": n / (t * 1e-3), "ms_per_call": t}
    side = torch.cuda.Stream(device=dev)
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        B.eig(dt, zt, rho, ws=ws, out=out, check=False)
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        B.eig(dt, zt, rho, ws=ws, out=out, check=False)
    g.replay()
    torch.cuda.synchronize()
    ms = []
    for _ in range(max(1, steps)):
        e0, e1 = _events()
        e0.record()
        for _ in range(reps):
            g.replay()
        e1.record()
        e1.synchronize()
        ms.append(e0.elapsed_time(e1) / reps)
    st = B.stream_status(ws)
    if st != 0:
        raise B.DPR1Error(st, "small")
    t = statistics.mean(ms)
    res["graph"] = {"value": n / (t * 1e-3), "ms_per_call": t}
    return res


def bench_accel(B, dev, d, z, rho, ws, out, flush, steps, bisection_ms):
    """The same workload with the accelerated bracketed solve (zero_finder = 1) in place of
    bisection: eigenpairs/s, phase times and evaluations of the secular function."""
    import torch
    n = d.numel()
    pe = B.PhaseEvents()
    opts = pe.attach(B.default_options(zero_finder=B.ACCELERATED))
    for _ in range(2):
        B.eig(d, z, rho, ws=ws, out=out, options=opts, check=False)
    torch.cuda.synchronize()
    st = B.stream_status(ws)
    if st != 0:
        raise B.DPR1Error(st, "accelerated warm-up")
    stats = B.workspace_stats(ws)
    ms, ph = [], []
    for _ in range(max(1, steps)):
        flush.zero_()
        e0, e1 = _events()
        e0.record()
        B.eig(d, z, rho, ws=ws, out=out, options=opts, check=False)
        e1.record()
        e1.synchronize()
        ms.append(e0.elapsed_time(e1))
        ph.append(pe.times_ms())
    st = B.stream_status(ws)
    if st != 0:
        raise B.DPR1Error(st, "accelerated timed")
    t = statistics.mean(ms)
    solve = statistics.mean(p[0] for p in ph)
    sh64, sh32 = shift_test_ops(n, stats)
    ops = ((n - 1) * (ACCEL_OPS_PER_TERM * stats["evals_solve"] + B64_OPS_PER_TERM * n
                      + DD_OPS_PER_TERM * stats["double_double"]) + sh64 + sh32 / FP32_PER_FP64
           + VEC_OPS_PER_ELEMENT * n * stats.get("tail_rows", 0))
    return {"zero_finder": "accelerated bracketed solve (nearest-pole rational model, value and slope)",
            "value": n / (t * 1e-3), "unit": "eigenpairs/s", "ms_per_step": t, "steps": len(ms),
            "phases_ms": {"solve": solve, "remedies": statistics.mean(p[1] for p in ph),
                          "eigenvectors": statistics.mean(p[2] for p in ph)},
            "evaluations": stats["evals_solve"], "evaluations_per_eigenpair": stats["evals_solve"] / n,
            "speedup_vs_bisection": bisection_ms / t,
            "solve_kernel_rate": {"achieved": ops / (solve * 1e-3) / 1e12, "unit": "T binary64-op-equivalent/s",
                                  "frac": ops / (solve * 1e-3) / NOMINAL_FP64_OPS,
                                  "ops_definition": "(n-1) x (8 ops per secular term and evaluation (5 for the "
                                                    "value, 3 for the slope) + per eigenvalue the 4-op binary64 "
                                                    "corner pass + 20 ops per double-double term where kappa_nu "
                                                    "asks for it) + the shift tests: per term 16 "
                                                    "binary32 ops of the binary32 pass, and 5 binary64 ops where "
                                                    "that pass leaves the sign open; the eigenvector rows its "
                                                    "lane groups write once its queue is empty, 6 binary64 ops "
                                                    "per component; a binary32 op counts 1/64"},
            "double_double_corners": stats["double_double"]}


def bench_hermitian(B, dev, n, seed, steps, flush):
    """The complex Hermitian D + rho z z^* (the hard spectrum with random phases on z):
    eigenvalues and the complex V (16 n^2 B), both zero finders."""
    import torch
    from paper_1405_7537_gb300 import workloads as W
    d, z, rho = W.hermitian(n, seed)
    dt = torch.tensor(d, device=dev)
    zt = torch.tensor(z, device=dev)
    ws = B.hermitian_workspace(n, dev)
    res = {"workload": "hard spectrum n=%d (seed %d) with phases exp(i theta), theta ~ U(0, 2 pi)" % (n, seed),
           "unit": "eigenpairs/s", "v_bytes": 16 * n * n}
    for name, zf in (("bisection", 0), ("accelerated", 1)):
        o = B.default_options(zero_finder=zf)
        B.eig_hermitian(dt, zt, rho, options=o, ws=ws)
        torch.cuda.synchronize()
        ms = []
        for _ in range(max(1, steps)):
            flush.zero_()
            e0, e1 = _events()
            e0.record()
            B.eig_hermitian(dt, zt, rho, options=o, ws=ws, check=False)
            e1.record()
            e1.synchronize()
            ms.append(e0.elapsed_time(e1))
        st = B.stream_status(ws)
        if st != 0:
            raise B.DPR1Error(st, "hermitian")
        t = statistics.mean(ms)
        res[name] = {"value": n / (t * 1e-3), "ms_per_step": t}
    return res


def bench_tridiag(B, dev, n, seed, steps):
    """Divide and conquer for a random symmetric tridiagonal matrix (every merge a DPR1 problem,
    each tree depth one batched launch), eigenvalues and eigenvectors, both zero finders;
    cuSOLVER's dense symmetric solver on the same matrix (torch.linalg.eigh) as context."""
    import torch
    from paper_1405_7537_gb300 import workloads as W
    a, b = W.tridiagonal(n, seed)
    at = torch.tensor(a, device=dev)
    bt = torch.tensor(b, device=dev)
    ws = B.tridiag_workspace(n, dev)
    T = 0
    while (1 << T) < n:
        T += 1
    # binary64 flops of the eigenvector products: 2 N (N1^2 + N2^2) per merge
    flops = 0
    for t in range(T):
        P = 1 << t
        for i in range(P):
            lo, hi = (i * n) >> t, ((i + 1) * n) >> t
            if hi - lo >= 2:
                mid = ((2 * i + 1) * n) >> (t + 1)
                flops += 2 * (hi - lo) * ((mid - lo) ** 2 + (hi - mid) ** 2)
    res = {"workload": "symmetric tridiagonal n=%d, a, b ~ U(-1, 1), seed %d; eigenvalues and Q" % (n, seed),
           "unit": "eigenpairs/s", "depths": T, "gemm_flops": flops}
    for name, zf in (("bisection", 0), ("accelerated", 1)):
        o = B.default_options(zero_finder=zf)
        B.eigh_tridiagonal(at, bt, options=o, ws=ws)
        torch.cuda.synchronize()
        ms = []
        for _ in range(max(1, steps)):
            e0, e1 = _events()
            e0.record()
            B.eigh_tridiagonal(at, bt, options=o, ws=ws, check=False)
            e1.record()
            e1.synchronize()
            ms.append(e0.elapsed_time(e1))
        st = B.stream_status(ws)
        if st != 0:
            raise B.DPR1Error(st, "tridiag")
        t = statistics.mean(ms)
        res[name] = {"value": n / (t * 1e-3), "ms_per_step": t}
    try:
        Td = torch.diag(at) + torch.diag(bt, 1) + torch.diag(bt, -1)
        torch.linalg.eigh(Td)
        torch.cuda.synchronize()
        e0, e1 = _events()
        e0.record()
        torch.linalg.eigh(Td)
        e1.record()
        e1.synchronize()
        ref_ms = e0.elapsed_time(e1)
        res["cusolver_dense_eigh"] = {"value": n / (ref_ms * 1e-3), "ms_per_step": ref_ms,
                                      "note": "torch.linalg.eigh on the dense n x n matrix (library, context only)"}
    except RuntimeError as e:            # torch's solver library may not load (e.g. under a profiler)
        res["cusolver_dense_eigh"] = {"unavailable": str(e).splitlines()[0]}
    return res


def bench_arrow(B, dev, n, seed, steps, flush):
    """The real symmetric arrowhead [D z; z^T alpha] of order n + 1 (d, z ~ U(-1, 1)): all
    eigenvalues and the (n+1)^2 eigenvector matrix with the K_nu remedies and the near-zero
    recompute, both zero finders; the counters of the last call show how many eigenvalues
    took which remedy."""
    import torch
    from paper_1405_7537_gb300 import workloads as W
    d, z, alpha = W.arrowhead(n, seed)
    dt = torch.tensor(np.array(d), device=dev)
    zt = torch.tensor(np.array(z), device=dev)
    ws = B.arrow_workspace(n, dev)
    res = {"workload": "arrowhead, n=%d poles (order n+1), d, z ~ U(-1, 1), alpha ~ U(-1, 1), seed %d" % (n, seed),
           "unit": "eigenpairs/s"}
    for name, zf in (("bisection", 0), ("accelerated", 1)):
        o = B.default_options(zero_finder=zf)
        B.eig_arrowhead(dt, zt, alpha, options=o, ws=ws)
        torch.cuda.synchronize()
        ms = []
        for _ in range(max(1, steps)):
            flush.zero_()
            e0, e1 = _events()
            e0.record()
            B.eig_arrowhead(dt, zt, alpha, options=o, ws=ws, check=False)
            e1.record()
            e1.synchronize()
            ms.append(e0.elapsed_time(e1))
        st = B.stream_status(ws)
        if st != 0:
            raise B.DPR1Error(st, "arrow")
        c = B.workspace_stats(ws)
        t = statistics.mean(ms)
        res[name] = {"value": (n + 1) / (t * 1e-3), "ms_per_step": t,
                     "remedies": {k: c[k] for k in ("flagged", "r1", "r2", "zero_path")}}
    return res


# ------------------------------------------------------------------ our arm
def kernel_source_hash(files):
    h = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_1405_7537_gb300", "csrc")
    for f in files:
        with open(os.path.join(csrc, f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def measured_hbm_gbs():
    """The measured HBM copy rate of this GPU type (MEASURED_PEAKS.json) and where it came from."""
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return float(json.load(f)["hbm_gbs"]), "of measured (MEASURED_PEAKS.json hbm_gbs)"
    except (OSError, ValueError, KeyError):
        return 6800.0, "of fallback (6.8 TB/s)"


def committed_traffic(n, zero_finder=0):
    """DRAM bytes per launch of the solve kernel from the committed ncu summary, if it was
    taken on the current kernel sources (else None).  The bisection's figure is a capture at
    its own order n (the stored elements of the inverse are re-read per evaluation, so the
    traffic does not scale with the eigenpair count); the accelerated solve's is per
    eigenpair (inputs read once, results written once) and scales with n."""
    path = os.path.join(ROOT, "profiles", "k_solve_traffic.json")
    try:
        with open(path) as f:
            rec = json.load(f)
    except (OSError, ValueError):
        return None
    try:
        if rec.get("source_hash") != kernel_source_hash(rec.get("source_files", [])):
            return None
    except OSError:
        return None
    ent = rec.get("accelerated" if zero_finder else "bisection", {})
    if "dram_bytes_per_eigenpair" in ent:
        return ent["dram_bytes_per_eigenpair"] * n
    if ent.get("n") == n:
        return ent.get("dram_bytes_per_launch")
    return None


def run_ours(args):
    import torch
    import torch.distributed as dist

    world, rank, local = dist_env()
    if world > 1:
        dist.init_process_group("nccl", init_method="env://")
    torch.cuda.set_device(local)
    from paper_1405_7537_gb300 import binding as B
    from paper_1405_7537_gb300 import workloads as W

    n = args.n
    d, z, rho = W.hard(n, SEED + rank)
    dev = torch.device("cuda", local)
    B.lib()
    dt_ = torch.tensor(np.array(d), device=dev)
    zt_ = torch.tensor(np.array(z), device=dev)
    ws = B.workspace(n, dev)
    out = dict(lam=torch.empty(n, dtype=torch.float64, device=dev),
               Vt=torch.empty((n, n), dtype=torch.float64, device=dev),
               sigma=torch.empty(n, dtype=torch.float64, device=dev),
               mu=torch.empty(n, dtype=torch.float64, device=dev),
               xnorm=torch.empty(n, dtype=torch.float64, device=dev))
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)
    pe = B.PhaseEvents()
    zf = args.zero_finder
    opts = pe.attach(B.default_options(zero_finder=zf))
    stream = torch.cuda.current_stream()

    def step():
        B.eig(dt_, zt_, rho, ws=ws, out=out, options=opts, check=False)

    # warm-up
    for _ in range(max(args.warmup, 0)):
        flush.zero_()
        step()
    torch.cuda.synchronize()
    st = B.stream_status(ws)
    if st != 0:
        raise B.DPR1Error(st, "bench warm-up")
    stats = B.workspace_stats(ws)

    # timed region
    sampler = ClockSampler(local)
    sampler.start()
    time.sleep(0.3)
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    step_ms, solve_ms, fix_ms, vec_ms = [], [], [], []
    t_wall0 = time.perf_counter()
    for _ in range(args.steps):
        flush.zero_()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        step()
        e1.record(stream)
        e1.synchronize()
        step_ms.append(e0.elapsed_time(e1))
        a, b, c = pe.times_ms()
        solve_ms.append(a); fix_ms.append(b); vec_ms.append(c)
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    wall = time.perf_counter() - t_wall0
    clocks = sampler.stop()
    value, total_ms = aggregate(sum(step_ms), n, args.steps, world, dist, dev)
    st = B.stream_status(ws)
    if st != 0:
        raise B.DPR1Error(st, "bench timed region")

    # roofline of the dominant kernel (the bisection kernel k_solve)
    evals = stats["evals_solve"]
    # bisection steps settled by a screen, decided by a certified bound or covered by the finishing step
    # take no binary64 evaluation; the screens' sums (bisection steps and probes) are binary32 work
    screened = stats.get("screened", 0)
    inferred = stats.get("inferred", 0)
    probes = stats.get("probes", 0)
    df = stats.get("screened_double_float", 0)
    n_dd = stats["double_double"]
    tail_rows = stats.get("tail_rows", 0)
    corner = B64_OPS_PER_TERM * n + DD_OPS_PER_TERM * n_dd
    ops32 = 0
    if zf == 0:
        b64_evals = evals - screened - inferred
        sh64, sh32 = shift_test_ops(n, stats)
        ops64 = (n - 1) * (OPS_PER_TERM * b64_evals + corner) + sh64 + VEC_OPS_PER_ELEMENT * n * tail_rows
        ops32 = (n - 1) * (B32_OPS_PER_TERM * max(screened + probes - df, 0) + DF_OPS_PER_TERM * df) + sh32
        kname = "k_solve (shift test, corner b, screened bisection)"
        odef = ("binary64: (n-1) x (5 ops (sub, fma, mul, div, add) per secular term x the bisection "
                "evaluations in binary64 + per eigenvalue the 4-op binary64 pass of the corner b (sub, "
                "div, mul, add) + for the eigenvalues whose kappa_nu asks for it 20 ops per double-double term "
                "of b (TwoSum 6, TwoProd 2, quotient and correction 5, compensated accumulation 7)); binary32: "
                "(n-1) x (14 ops per term of a binary32 screen + 50 per term of a double-float screen) over the "
                "settled screens of bisection steps and probes; the shift tests: per term 16 "
                "binary32 ops of the binary32 pass, and the 5-op binary64 pass where the binary32 pass leaves "
                "the sign open; the eigenvector rows written by the kernel's lane groups once its queue is "
                "empty, 6 binary64 ops per component; a binary32 op counts 1/64 of a binary64 op (128 against "
                "2 lanes per SM and clock); steps decided by certified bounds are not counted")
    else:
        b64_evals = evals
        sh64, sh32 = shift_test_ops(n, stats)
        ops64 = (n - 1) * (ACCEL_OPS_PER_TERM * evals + corner) + sh64 + VEC_OPS_PER_ELEMENT * n * tail_rows
        ops32 = sh32
        kname = "k_solve (shift test, corner b, accelerated bracketed solve)"
        odef = ("(n-1) x (8 ops per secular term and evaluation (5 for the value, 3 for the slope) + per "
                "eigenvalue the 4-op binary64 corner pass + 20 ops per double-double term for the eigenvalues "
                "whose kappa_nu asks for it) + the shift tests: per term 16 binary32 ops of "
                "the binary32 pass, and 5 binary64 ops where it leaves the sign open; the eigenvector rows "
                "written by its lane groups once its queue is empty, 6 binary64 ops per component; a binary32 "
                "op counts 1/64")
    ops = ops64 + ops32 / FP32_PER_FP64
    t_solve = statistics.mean(solve_ms) * 1e-3
    achieved = ops / t_solve
    # live binary64 fma rate of this GPU at this clock (same process, after the timed region)
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    sink = torch.empty(sms * 4 * 256, dtype=torch.float64, device=dev)
    B.probe_dfma(sms * 4, 256, 64, sink)
    torch.cuda.synchronize()
    pe0 = torch.cuda.Event(enable_timing=True); pe1 = torch.cuda.Event(enable_timing=True)
    pe0.record(stream)
    B.probe_dfma(sms * 4, 256, 4096, sink)
    pe1.record(stream)
    pe1.synchronize()
    measured_fma = sms * 4 * 256 * 4096 * 8 / (pe0.elapsed_time(pe1) * 1e-3)
    roof = {"bound": "alu", "kernel": kname,
            "achieved": achieved / 1e12, "peak": NOMINAL_FP64_OPS / 1e12,
            "unit": "T binary64-op-equivalent/s",
            "frac": achieved / NOMINAL_FP64_OPS, "traffic": committed_traffic(n, zf),
            "peak_source": "nominal GB300 binary64 1.25 TFLOP/s = 2 fma/clk/SM x 152 SMs x 2070 MHz "
                           "(MEASURED_PEAKS.json has no binary64 entry)",
            "measured_fma_rate": measured_fma / 1e12,
            "frac_of_measured_fma_rate": achieved / measured_fma,
            "ops_per_launch": ops, "ops_definition": odef,
            "binary64_ops": ops64, "binary32_ops": ops32,
            "binary64_frac": ops64 / t_solve / NOMINAL_FP64_OPS,
            "binary32_frac": ops32 / t_solve / (FP32_PER_FP64 * NOMINAL_FP64_OPS),
            "launch_ms": 1e3 * t_solve, "bisection_steps": evals,
            "binary64_evaluations": b64_evals, "screened_steps": screened, "inferred_steps": inferred,
            "screened_probes": probes, "double_float_settled": df, "double_double_corners": n_dd,
            "shift_tests_binary32": stats.get("shift_binary32", 0),
            "eigenvector_rows_written": tail_rows,
            # the plain bisection's terms (every step and the shift-test pass) per second
            # secular terms per second in the passes that ran: evaluations, screens, shift tests
            "term_rate": (n - 1) * (b64_evals + screened + probes + n) / t_solve}

    # the eigenvector phase (k_vectors and the short near-zero and deflation kernels before it):
    # the n^2 write of V against the measured copy rate, and its binary64 work against the peak
    t_vec = statistics.mean(vec_ms) * 1e-3
    hbm_peak = measured_hbm_gbs()
    # the rows k_vectors writes: those the solve kernel's tail did not, and the tail's rows whose
    # pair the remedies changed
    vec_rows = stats.get("vector_rows", n - tail_rows)
    v_bytes = 8.0 * n * vec_rows
    v_ops = float(VEC_OPS_PER_ELEMENT) * n * vec_rows
    hbm_frac = v_bytes / t_vec / (hbm_peak[0] * 1e9)
    alu_frac = v_ops / t_vec / NOMINAL_FP64_OPS
    phase_roofs = {"eigenvectors": {
        "bound": "alu" if alu_frac >= hbm_frac else "hbm", "ms": 1e3 * t_vec,
        "hbm": {"achieved": v_bytes / t_vec / 1e9, "peak": hbm_peak[0], "unit": "GB/s", "frac": hbm_frac,
                "peak_source": hbm_peak[1], "rows": vec_rows,
                "bytes_definition": "8 n bytes per row of V that k_vectors writes, once"},
        "alu": {"achieved": v_ops / t_vec / 1e12, "peak": NOMINAL_FP64_OPS / 1e12, "unit": "T binary64-op/s",
                "frac": alu_frac, "ops_definition": "per element: 2 sub, 1 div, 1 mul, 1 fma (sum of squares), "
                                                    "1 mul (rescale)"}}}

    # end to end through the public API with host buffers
    e2e = None
    if args.e2e_steps > 0:
        d_h = torch.from_numpy(np.array(d)).pin_memory()
        z_h = torch.from_numpy(np.array(z)).pin_memory()
        lam_h = torch.empty(n, dtype=torch.float64).pin_memory()
        sig_h = torch.empty(n, dtype=torch.float64).pin_memory()
        mu_h = torch.empty(n, dtype=torch.float64).pin_memory()
        Vt_h = torch.empty((n, n), dtype=torch.float64).pin_memory()

        e2e_opts = B.default_options(zero_finder=zf)
        # double-buffered outputs: step t computes into buffer t % 2 on the compute stream while
        # a copy stream reads step t - 1's results back to the host
        f64 = dict(dtype=torch.float64, device=dev)
        outs = [out, dict(lam=torch.empty(n, **f64), Vt=torch.empty((n, n), **f64), sigma=torch.empty(n, **f64),
                          mu=torch.empty(n, **f64), xnorm=torch.empty(n, **f64))]
        copy_stream = torch.cuda.Stream(device=dev)
        copied = [torch.cuda.Event(), torch.cuda.Event()]
        for e in copied:
            e.record(copy_stream)

        def e2e_step(t):
            b = t % 2
            flush.zero_()
            stream.wait_event(copied[b])          # the host copy of this buffer's last contents is done
            r = B.eig(d_h, z_h, rho, ws=ws, out=outs[b], options=e2e_opts, check=False, stream=stream)
            ready = torch.cuda.Event()
            ready.record(stream)
            copy_stream.wait_event(ready)
            with torch.cuda.stream(copy_stream):
                lam_h.copy_(r["lam"], non_blocking=True)
                sig_h.copy_(r["sigma"], non_blocking=True)
                mu_h.copy_(r["mu"], non_blocking=True)
                Vt_h.copy_(r["Vt"], non_blocking=True)
            copied[b].record(copy_stream)

        e2e_step(0)
        e2e_step(1)
        torch.cuda.synchronize()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for t in range(args.e2e_steps):
            e2e_step(t)
        stream.wait_stream(copy_stream)
        e1.record(stream)
        e1.synchronize()
        st = B.stream_status(ws)
        if st != 0:
            raise B.DPR1Error(st, "bench end to end")
        e2e_value, e2e_ms = aggregate(e0.elapsed_time(e1), n, args.e2e_steps, world, dist, dev)
        e2e = {"value": e2e_value, "unit": "eigenpairs/s",
               "h2d_bytes_per_step": 2 * 8 * n, "d2h_bytes_per_step": 3 * 8 * n + 8 * n * n,
               "ms_per_step": e2e_ms / args.e2e_steps, "steps": args.e2e_steps,
               "pipelining": "two device output sets: the device-to-host copy of step t (lambda, sigma, mu, V) "
                             "overlaps the compute of step t + 1; every step copies its own inputs in and "
                             "its results out"}

    extras = {}
    which = set() if args.no_extras else set(x.strip() for x in args.extras.split(",") if x.strip())
    if "small" in which:
        extras["small"] = bench_small(B, dev, 3)
    if "fwd_bwd" in which:
        extras["fwd_bwd"] = bench_fwd_bwd(B, dev, 4096, 2, 3, True)
    if "fwd_bwd_large" in which:
        extras["fwd_bwd_large"] = bench_fwd_bwd(B, dev, 32768, 4, 2, False)
    if "batched" in which:
        extras["batched"] = bench_batched(B, dev, 2)
    if "arrow" in which:
        extras["arrow"] = bench_arrow(B, dev, n, 6, 2, flush)
    if "tridiag" in which:
        extras["tridiag"] = bench_tridiag(B, dev, 4096, 5, 3)
    if "hermitian" in which:
        extras["hermitian"] = bench_hermitian(B, dev, n, SEED, 2, flush)
    if "accel" in which:
        extras["accelerated"] = bench_accel(B, dev, dt_, zt_, rho, ws, out, flush, 3, total_ms / args.steps / world)

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        rate, threads, m, dtc = cpu_oracle_rate(d, z, rho, args.cpu_sample)
        rate1, _, m1, dt1 = cpu_oracle_rate(d, z, rho, max(16, args.cpu_sample // 32), seed=8, threads=1)
        cpu = {"value": rate, "unit": "eigenpairs/s", "cores": threads, "kind": "oracle",
               "sample": "%d random eigenpairs of the same n=%d workload (%.1f s wall on %d threads)"
                         % (m, n, dtc, threads),
               "single_thread": {"value": rate1, "unit": "eigenpairs/s", "cores": 1,
                                 "sample": "%d random eigenpairs of the same workload (%.1f s wall)" % (m1, dt1)}}

    if rank == 0:
        line = {"metric": METRIC, "value": value, "unit": "eigenpairs/s", "n_gpus": world, "steps": args.steps,
                "warmup": args.warmup, "ms_per_step": total_ms / args.steps, "higher_is_better": True,
                "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
                "config": dict(workload_config(n), zero_finder=("bisection" if zf == 0 else "accelerated")),
                "roofline": roof, "phase_rooflines": phase_roofs, "cpu_baseline": cpu, "e2e": e2e,
                "gpu_launches": LAUNCHES_PER_CALL * args.steps, "clocks": clocks,
                "phases_ms": {"bisection": statistics.mean(solve_ms), "remedies": statistics.mean(fix_ms),
                              "eigenvectors": statistics.mean(vec_ms)},
                "remedy_counts": {"flagged": stats["flagged"], "r1": stats["r1"], "r2": stats["r2"],
                                  "zero_path": stats["zero_path"]},
                "wall_s_timed_region": wall}
        line.update(extras)
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()
    return 0


def run_only(args):
    """One extra measurement alone (used for small ncu captures of its kernels)."""
    import torch
    torch.cuda.set_device(0)
    from paper_1405_7537_gb300 import binding as B
    dev = torch.device("cuda", 0)
    B.lib()
    if args.only == "tridiag":
        res = bench_tridiag(B, dev, args.n, 5, args.steps)
    elif args.only == "hermitian":
        flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)
        res = bench_hermitian(B, dev, args.n, SEED, args.steps, flush)
    elif args.only == "arrow":
        flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)
        res = bench_arrow(B, dev, args.n, 6, args.steps, flush)
    else:
        res = bench_fwd_bwd(B, dev, args.n, 2, args.steps, True)
    print(json.dumps({"only": args.only, "n": args.n, args.only: res}), flush=True)
    return 0


def main():
    args = parse()
    if args.impl == "reference":
        return run_reference(args)
    if args.only:
        return run_only(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
