#!/usr/bin/env python
"""Benchmark: simplex iterations/s and time-to-optimum of the FP64 dense
revised simplex on the dense real 4096 x 8192 workload (A_ij ~ U[0,1) with 10%
zeros, b_i ~ U[n/4, n/2], c_j ~ U[0,1), seed 1; reinversion every 64 pivots,
tabu tenure 7).

One step = one full solve from the slack basis to optimality (every row of
the hot path: PRICE+CHUZC, UPDATE+FTRAN+CHUZR, pivot bookkeeping, periodic
reinversion), with A, b, c already resident in HBM.  value = pivots / second
over the K timed steps.  The per-iteration working set (A 268 MB + B^-1 134
MB) is larger than L2, so no flush is needed between iterations.

  python bench.py [--gpus N --steps K --warmup W] [--impl reference]

N > 1 (torchrun): every rank solves its own replica (the method has no
data-parallel exchange on one LP); value = all ranks' pivots / max time.
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
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "simplex iters/s & time-to-optimum, m=4096 n=8192 FP64; batched LPs/s"
WORKLOAD = dict(name="dense_real_4096x8192", kind="real", m=4096, n=8192, seed=1)


def _dist():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled every 200 ms."""

    FIELDS = ["clocks.sm", "clocks.max.sm", "power.draw", "clocks_event_reasons.hw_slowdown",
              "clocks_event_reasons.hw_thermal_slowdown", "clocks_event_reasons.sw_thermal_slowdown",
              "clocks_event_reasons.sw_power_cap"]

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []
        self.thread = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), "--query-gpu=" + ",".join(self.FIELDS),
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
            return
        self.thread = threading.Thread(target=self._read, daemon=True)
        self.thread.start()

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append((time.time(), line.strip()))

    def stop(self, t0: float, t1: float) -> dict:
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        if self.thread:
            self.thread.join(timeout=2)
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ts, line in self.lines:
            if ts < t0 - 0.25 or ts > t1 + 0.25:
                continue
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 7:
                continue
            try:
                sm.append(float(parts[0]))
                smax.append(float(parts[1]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[3:7]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(smax) if smax else None,
                "samples": len(sm), "reasons": sorted(reasons)}


def _peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return float(d.get("hbm_gbs", 6800.0)), "measured"
    return 6800.0, "fallback"


# FP64 peak of the GB300: 1.25 TFLOP/s nominal, i.e. 2 FP64 FMA per clock per
# SM x 152 SMs x 2.07 GHz x 2 flops (no FP64 figure is among the measured
# peaks; a standalone FMA-chain probe reached 1.20 TFLOP/s, 96% of it).
FP64_PEAK_TFLOPS = 1.25
# Kernel durations come from CUDA events around the PRICE and UPDATE launches
# of one pivot (the first) of each 64-pivot captured graph, inside the timed
# solves; the other pivots keep their launch overlap.
KERNEL_TIMING_STRIDE = 64


def _traffic(kernel: str):
    """dram bytes per launch from the committed ncu capture, if the kernel's
    source has not changed since."""
    p = os.path.join(ROOT, "profiles", "ncu_traffic.json")
    if not os.path.exists(p):
        return None
    d = json.load(open(p))
    ent = d.get(kernel)
    if not ent:
        return None
    src = os.path.join(ROOT, "paper_1803_04378_gb300", "csrc", ent["source"])
    if not os.path.exists(src):
        return None
    sha = hashlib.sha256(open(src, "rb").read()).hexdigest()[:16]
    if sha != ent.get("source_sha"):
        return None
    return ent.get("dram_bytes_per_launch_full_size")


def _oracle_golden():
    """The oracle's full solve of the timed workload (objective, pivot count),
    stored by tests/golden/make_fullsize.py, which calls only the oracle."""
    p = os.path.join(ROOT, "tests", "golden", f"{WORKLOAD['name']}.json")
    if not os.path.exists(p):
        return None
    with open(p) as f:
        return json.load(f)


def _rel_err(z, ref):
    return None if ref is None else abs(z - ref) / max(1.0, abs(ref))


def _certificate(A, b, c, x, y):
    """Optimality residuals of the returned solution (host, numpy): primal
    infeasibility of Ax <= b, x >= 0 and dual infeasibility of A^T y >= c,
    y >= 0, relative to max|b| and max|c|, and the relative duality gap."""
    import numpy as np
    x = np.asarray(x, dtype=np.float64)
    y = np.asarray(y, dtype=np.float64)
    s = b - A @ x
    primal = max(float(np.max(-s, initial=0.0)), float(np.max(-x, initial=0.0)))
    dual = max(float(np.max(c - A.T @ y, initial=0.0)), float(np.max(-y, initial=0.0)))
    pz, dz = float(c @ x), float(b @ y)
    return {"primal_residual": primal / max(1.0, float(np.max(np.abs(b)))) + 0.0,
            "dual_residual": dual / max(1.0, float(np.max(np.abs(c)))),
            "gap_rel": abs(pz - dz) / max(1.0, abs(pz))}


def oracle_sample(A, b, c, iters: int, threads: int):
    """One timed oracle run over the first `iters` pivots from the slack basis
    (with iters >= 64 the reinversion after pivot 64 is included); returns
    (pivots, seconds)."""
    import oracle
    t0 = time.perf_counter()
    s = oracle.solve(A, b, c, oracle.Options(max_iters=iters), threads=threads)
    return s.iterations, time.perf_counter() - t0


def cpu_baseline(A, b, c, iters: int):
    """The oracle (plain C, unmodified) on the first `iters` pivots of the
    same workload, the reinversion after pivot 64 included: the serial build
    (the paper's sequential version) and the OpenMP build on every host core
    (bit-identical results; PRICE columns, FTRAN and update rows and the
    elimination rows shared among threads)."""
    import oracle
    its, dt = oracle_sample(A, b, c, iters, 1)
    out = {"value": its / dt, "unit": "iters/s", "cores": 1, "kind": "oracle",
           "sample": f"first {its} pivots of {WORKLOAD['name']} from the slack basis, the reinversion after "
                     f"pivot 64 included (single-threaded plain C FP64 revised simplex), {dt:.1f} s"}
    nt = oracle.threads_used(0)
    its_p, dt_p = oracle_sample(A, b, c, iters, 0)
    out["all_cores"] = {"value": its_p / dt_p, "unit": "iters/s", "cores": nt, "kind": "oracle (OpenMP build)",
                        "sample": f"the same {its_p} pivots, {dt_p:.1f} s"}
    return out


def run_batched(lpgb, args, with_cpu: bool):
    """4096 independent dense integer LPs (m uniform 16..256, n uniform
    m..2m, each generated like the 200x200 dense integer workload) solved in
    persistent launches; per-bucket launch configuration from the autotuner."""
    import numpy as np
    import lpgen
    count = args.batch_count
    ms, ns = lpgen.batch_sizes(count, seed=3)
    probs = [lpgen.batch_lp(k, int(ms[k]), int(ns[k])) for k in range(count)]
    with lpgb.Batch(probs) as bt:
        table = bt.tune(trials=1)
        for _ in range(max(1, args.warmup)):
            bt.solve()
        secs, its, fl = 0.0, 0, 0.0
        steps = max(1, args.steps)
        for _ in range(steps):
            r = bt.solve()
            secs += r["seconds"]
            its += r["iterations"]
            fl += r["fp64_flops"]
        st, it, obj, xs, ys = bt.results()
        solved = int(np.sum(st == 1))
    out = {"metric": "batched LPs/s", "value": count * steps / secs, "unit": "LPs/s",
           "config": {"workload": "batch_4096_small", "count": count, "m": "uniform 16..256",
                      "n": "uniform m..2m", "price": "BF16 screen, top 8 re-priced in FP64",
                      "tuning": [int(v) for v in table]},
           "seconds_per_batch": secs / steps, "pivots_per_batch": its // steps, "solved": solved,
           "roofline": {"bound": "alu", "unit": "TFLOP/s", "achieved": fl / secs / 1e12,
                        "peak": FP64_PEAK_TFLOPS, "frac": None,
                        "what": "FP64 flops that FTRAN, the update and the re-price of the dense B^-1 would "
                                "take; the solver leaves out the exact zeros of its unit columns, so the "
                                "rate passes the pipe's and has no fraction of it"}}
    # the plain single-LP GPU solver on a sample of the same LPs (one handle
    # per LP, FP64 PRICE, device solve time only)
    sample, t_plain, gap = 64, 0.0, 0.0
    for k in range(min(sample, count)):
        with lpgb.LP(*probs[k]) as lp1:
            r1 = lp1.solve()
            z1 = lp1.solution()[2]
        t_plain += r1.seconds
        gap = max(gap, abs(z1 - float(obj[k])) / max(1.0, abs(z1)))
    out["plain_gpu_solver"] = {"value": min(sample, count) / t_plain, "unit": "LPs/s",
                               "sample": f"first {min(sample, count)} LPs of the batch, one lp_solve each",
                               "batched_speedup": out["value"] / (min(sample, count) / t_plain),
                               "max_rel_objective_gap_vs_batched": gap}
    if with_cpu:
        import oracle
        sample = 32
        t0 = time.perf_counter()
        sols = [oracle.solve(*probs[k]) for k in range(sample)]
        dt = time.perf_counter() - t0
        out["cpu_baseline"] = {"value": sample / dt, "unit": "LPs/s", "cores": 1, "kind": "oracle",
                               "sample": f"first {sample} LPs of the batch, single-threaded oracle, {dt:.1f} s"}
        out["max_objective_rel_err_vs_oracle"] = max(
            abs(float(obj[k]) - s_.objective) / max(1.0, abs(s_.objective)) for k, s_ in enumerate(sols))
        out["status_equal_oracle"] = all(int(st[k]) == s_.status for k, s_ in enumerate(sols))
        out["oracle_checked_lps"] = sample
    return out


def aggregate_ranks(elapsed: float, iters: int, ws: int, device):
    """Whole-job figures of N replicas: the slowest rank's time and the pivots
    of all ranks (value = their ratio).  Needs an initialised process group
    when ws > 1 (NCCL on the GPUs, gloo in the CPU tests)."""
    if ws <= 1:
        return elapsed, iters
    import torch
    import torch.distributed as dist
    tt = torch.tensor([elapsed], dtype=torch.float64, device=device)
    dist.all_reduce(tt, op=dist.ReduceOp.MAX)
    it_t = torch.tensor([iters], dtype=torch.int64, device=device)
    dist.all_reduce(it_t)
    return float(tt.item()), int(it_t.item())


def run_reference(args):
    ws, rank, local = _dist()
    if rank != 0:
        return 0
    import lpgen
    import oracle
    A, b, c = lpgen.make(WORKLOAD["kind"], WORKLOAD["m"], WORKLOAD["n"], WORKLOAD["seed"])
    oracle.build()
    # the same sample as cpu_baseline (first 64 pivots, the reinversion after
    # pivot 64 included); each timed step is one run of it.  Warm-up runs are
    # capped at one: the oracle has no caches to warm beyond the first run.
    sample = args.cpu_iters
    times = []
    for step in range(min(1, args.warmup) + args.steps):
        its, dt = oracle_sample(A, b, c, sample, 1)
        if step >= min(1, args.warmup):
            times.append(dt)
    total = sum(times)
    value = its * len(times) / total
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": "iters/s",
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * total / len(times), "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": WORKLOAD["name"], "m": WORKLOAD["m"], "n": WORKLOAD["n"],
                       "seed": WORKLOAD["seed"], "A": "U[0,1) with 10% zeros", "reinvert_every": 64,
                       "tabu_tenure": 7,
                       "step": f"first {its} pivots from the slack basis"
                               + (" (the reinversion after pivot 64 included)" if its >= 64 else "")},
            "cpu_baseline": {"value": value, "unit": "iters/s", "cores": 1, "kind": "oracle",
                             "sample": f"first {its} pivots of {WORKLOAD['name']} per step, "
                                       f"the same sample as the GPU line's cpu_baseline"},
            "e2e": {"value": value, "unit": "iters/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


def run_warmstart(lpgb):
    """Pattern (4), reduced so that the bench stays within minutes: the learned
    warm start on the family of its configured run (m = 1024, n = 2048, base
    as the dense real workload with seed 4, every entry times N(1, 0.05^2))
    with 2000 label solves instead of 20000, the proposal threshold picked on
    50 validation instances, and 100 held-out instances solved cold and from
    the repaired proposal.  The configured run (20000 / 1000) is
    `python -m paper_1803_04378_gb300.warmstart`."""
    import lpgen
    from paper_1803_04378_gb300 import warmstart as wsm
    base = lpgen.dense_real_lp(1024, 2048, 4)
    fam = wsm.Family(base)
    t0 = time.perf_counter()
    X, Y, piv = wsm.generate_labels(fam, range(1, 2001))
    t_labels = time.perf_counter() - t0
    net, losses = wsm.train(X, Y, epochs=20)
    sel = {}
    for t in (1.0, 2.0, 3.0):
        sv = wsm.summarize(wsm.evaluate(fam, net, range(30_000_000, 30_000_050), ("repair",), None, t), ("repair",))
        sel[t] = sv["repair"]["speedup"]
    thr = max(sel, key=sel.get)
    rows = wsm.evaluate(fam, net, range(10_000_000, 10_000_100), ("repair",), None, thr)
    sm = wsm.summarize(rows, ("repair",))
    fam.close()
    net.close()
    r = sm["repair"]
    return {"value": r["speedup"], "unit": "x (cold / warm time-to-optimum)",
            "cold_time_to_optimum_s": sm["cold_time_to_optimum_s"], "warm_time_to_optimum_s": r["time_to_optimum_s"],
            "cold_pivots_mean": sm["cold_pivots_mean"], "warm_pivots_mean": r["pivots_mean"],
            "repair_pivots_mean": r["repairs_mean"], "faster_fraction": r["faster_fraction"],
            "max_rel_objective_gap_vs_cold": r["max_rel_objective_gap"], "all_optimal": r["optimal"],
            "threshold": thr, "validation_speedups": sel, "label_seconds": t_labels,
            "what": ("learned warm start on the 1024 x 2048 family: 2000 training pairs (the configured run "
                     "uses 20000), 100 held-out instances, inference on the device included")}


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--cpu-iters", type=int, default=64,
                    help="pivots of the CPU baseline sample (64: the reinversion after pivot 64 included)")
    ap.add_argument("--e2e-steps", type=int, default=3)
    ap.add_argument("--skip-cpu", action="store_true")
    ap.add_argument("--skip-variants", action="store_true")
    ap.add_argument("--skip-batch", action="store_true")
    ap.add_argument("--skip-warmstart", action="store_true")
    ap.add_argument("--price-mode", type=int, default=0, help="PRICE of the timed solves (profiling)")
    ap.add_argument("--engine", type=int, default=2,
                    help="LP_ENGINE_* of the timed solves: 0 dense persistent, 1 graphs, 2 slack-structured")
    ap.add_argument("--batch-count", type=int, default=4096)
    ap.add_argument("--only-batch", action="store_true", help="run only the batched leg (profiling)")
    ap.add_argument("--reinversion-only", type=int, default=0,
                    help="profiling: solve once, then time this many reinversions of the optimal basis")
    ap.add_argument("--graph-iters", type=int, default=0,
                    help="pivots per persistent launch or captured graph (profiling; default 64)")
    ap.add_argument("--reinvert-every", type=int, default=-1,
                    help="profiling: pivots between reinversions (0: none; default: the solver's 64)")
    ap.add_argument("--max-iters", type=int, default=0,
                    help="stop every solve after this many pivots (profiling runs only)")
    args = ap.parse_args()
    if args.warmup < 3:
        print("warning: fewer than 3 warm-up steps", file=sys.stderr)
    if args.impl == "reference":
        return run_reference(args)

    import numpy as np
    import torch

    import lpgen
    ws, rank, local = _dist()
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    torch.cuda.set_device(local)
    from paper_1803_04378_gb300 import build as _build
    _build.build()
    from paper_1803_04378_gb300 import lpgb

    if args.only_batch:
        print(json.dumps(run_batched(lpgb, args, False)), flush=True)
        return 0
    m, n = WORKLOAD["m"], WORKLOAD["n"]
    A, b, c = lpgen.make(WORKLOAD["kind"], m, n, WORKLOAD["seed"])
    stream = torch.cuda.current_stream()
    At, bt, ct = (torch.from_numpy(v).cuda() for v in (A, b, c))
    extra = {"max_iters": args.max_iters} if args.max_iters > 0 else {}
    if args.graph_iters > 0:
        extra["graph_iters"] = args.graph_iters
    extra["engine"] = args.engine
    if args.reinvert_every >= 0:
        extra["reinvert_every"] = args.reinvert_every
    lp = lpgb.LP(At, bt, ct, kernel_timing=KERNEL_TIMING_STRIDE, cuda_stream=stream.cuda_stream, price_mode=args.price_mode, **extra)
    del At, bt, ct

    def barrier():
        if ws > 1:
            torch.distributed.barrier()

    if args.reinversion_only > 0:
        lp.solve()
        basis = lp.basis()
        k = int(sum(1 for v in basis if v < n))
        with lpgb.LP(torch.from_numpy(A).cuda(), torch.from_numpy(b).cuda(), torch.from_numpy(c).cuda(),
                     max_iters=0) as lr:
            times = []
            for _ in range(args.reinversion_only):
                lr.set_basis(basis)
                r = lr.solve()
                times.append((r.reinvert_seconds, r.reinvert_gj_seconds, r.reinvert_assemble_seconds))
        t = np.array(times)
        print(json.dumps({"reinversion_of_optimal_basis": {"k_structural": k, "m": m,
                                                           "seconds_mean": float(t[:, 0].mean()),
                                                           "gj_seconds_mean": float(t[:, 1].mean()),
                                                           "assemble_seconds_mean": float(t[:, 2].mean())}}))
        lp.close()
        return 0

    for _ in range(args.warmup):
        lp.reset()
        lp.solve()

    sampler = ClockSampler(local)
    sampler.start()
    time.sleep(0.5)
    barrier()
    torch.cuda.synchronize()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    t_wall0 = time.time()
    e0.record(stream)
    results = []
    for _ in range(args.steps):
        lp.reset()
        results.append(lp.solve())
    e1.record(stream)
    torch.cuda.synchronize()
    barrier()
    t_wall1 = time.time()
    clocks = sampler.stop(t_wall0, t_wall1)
    elapsed = e0.elapsed_time(e1) * 1e-3
    iters = sum(r.iterations for r in results)
    x, y, z = lp.solution()
    elapsed, iters_all = aggregate_ranks(elapsed, iters, ws, "cuda")

    # dominant kernel and its live roofline
    ps = sum(r.price_seconds for r in results)
    us = sum(r.update_seconds for r in results)
    pn = sum(r.price_launches for r in results)
    un = sum(r.update_launches for r in results)
    pb = sum(r.price_bytes for r in results)
    ub = sum(r.update_bytes for r in results)
    cs = sum(r.chain_seconds for r in results)
    cn = sum(r.chain_launches for r in results)
    cb = sum(r.chain_bytes for r in results)
    if cn > 0:
        # persistent engine: every launch runs PRICE + UPDATE/FTRAN of up to 64
        # pivots; both do one FP64 FMA per 8 algorithmic bytes
        kname = "k_iterate_r" if results[0].persistent == 2 else "k_iterate"
        kt, kn, kb, kflops = cs, cn, cb, cb / 4.0
    elif us >= ps:
        kname, kt, kn, kb, kflops = "k_update", us, un, ub, 4.0 * m * m * un
    else:
        kname, kt, kn, kb, kflops = "k_price", ps, pn, pb, 2.0 * pb / 8.0
    hbm_peak, peak_kind = _peaks()
    achieved = (kb / kn) / (kt / kn) / 1e9 if kn else None
    hbm = {"achieved": achieved, "peak": hbm_peak, "unit": "GB/s",
           "frac": (achieved / hbm_peak) if achieved else None, "peak_source": f"{peak_kind} hbm_gbs"}
    fp64 = {"achieved": kflops / kt / 1e12 if kt else None, "peak": FP64_PEAK_TFLOPS, "unit": "TFLOP/s",
            "frac": (kflops / kt / 1e12 / FP64_PEAK_TFLOPS) if kt else None,
            "peak_source": "nominal FP64 rate (2 FMA per clock per SM x 152 SMs x 2.07 GHz), no measured FP64 peak"}
    if kname == "k_iterate_r":
        # the live rows of A and columns of B^-1 stay in shared memory (where they fit,
        # else in L2) across pivots: the bound is the FP64 pipe, and the HBM figure
        # is given beside it
        roofline = dict(bound="alu", kernel=kname, **fp64, hbm=hbm)
    else:
        roofline = dict(bound="hbm", kernel=kname, **hbm, fp64=fp64)
    roofline.update({"traffic": _traffic(kname),
                     "bytes_per_launch": kb / kn if kn else None,
                     "flops_per_launch": kflops / kn if kn else None,
                     "avg_launch_us": 1e6 * kt / kn if kn else None,
                     "share_of_step": kt / sum(r.seconds for r in results)})
    chain_bytes = sum(r.bytes_moved for r in results)
    reinv_s = sum(r.reinvert_seconds for r in results)
    iter_s = sum(r.seconds for r in results) - reinv_s

    # end to end through the public API with host (pinned) buffers
    e2e = None
    if args.e2e_steps > 0:
        Ap = torch.empty((m, n), dtype=torch.float64, pin_memory=True)
        bp = torch.empty(m, dtype=torch.float64, pin_memory=True)
        cp = torch.empty(n, dtype=torch.float64, pin_memory=True)
        Ap.numpy()[:] = A
        bp.numpy()[:] = b
        cp.numpy()[:] = c
        it_e2e, t_e2e = 0, 0.0
        for _ in range(args.e2e_steps):
            torch.cuda.synchronize()
            barrier()
            t0 = time.perf_counter()
            with lpgb.LP(Ap.numpy(), bp.numpy(), cp.numpy(), cuda_stream=stream.cuda_stream, **extra) as lp2:
                r2 = lp2.solve()
                x2, y2, z2 = lp2.solution()
            torch.cuda.synchronize()
            t_e2e += time.perf_counter() - t0
            it_e2e += r2.iterations
        e2e = {"value": it_e2e / t_e2e, "unit": "iters/s",
               "h2d_bytes_per_step": 8 * (m * n + m + n), "d2h_bytes_per_step": 8 * (n + m) + 8,
               "seconds_per_step": t_e2e / args.e2e_steps}

    golden = _oracle_golden()
    z_oracle = golden["objective"] if golden else None

    # variant: BF16-screened PRICE, each screening block's best two columns
    # re-priced in FP64 (same FP64 UPDATE/FTRAN/ratio test/reinversion;
    # optimality certified in FP64)
    variants = {}
    if not args.skip_variants:
        # variant: the other persistent engine (same pivots): the dense m x m
        # inverse when the structured one is timed, and the reverse
        other = 0 if args.engine == 2 else 2
        At, bt, ct = (torch.from_numpy(v).cuda() for v in (A, b, c))
        xs = dict(extra, engine=other)
        with lpgb.LP(At, bt, ct, kernel_timing=KERNEL_TIMING_STRIDE, cuda_stream=stream.cuda_stream, **xs) as lps:
            del At, bt, ct
            lps.solve()  # warm-up
            lps.reset()
            torch.cuda.synchronize()
            v0 = torch.cuda.Event(enable_timing=True)
            v1 = torch.cuda.Event(enable_timing=True)
            v0.record(stream)
            rs_ = lps.solve()
            v1.record(stream)
            torch.cuda.synchronize()
            ts_ = v0.elapsed_time(v1) * 1e-3
            zs_ = lps.solution()[2]
        variants["dense_engine" if other == 0 else "structured_engine"] = {
            "value": rs_.iterations / ts_, "unit": "iters/s", "time_to_optimum_s": ts_,
            "pivots_per_solve": rs_.iterations, "reinversions_per_solve": rs_.reinversions,
            "objective": zs_, "objective_rel_err_vs_timed_engine": abs(zs_ - z) / max(1.0, abs(z)),
            "objective_rel_err_vs_oracle": _rel_err(zs_, z_oracle),
            "reinversion_seconds": rs_.reinvert_seconds,
            "us_per_pivot_excl_reinversion": 1e6 * (ts_ - rs_.reinvert_seconds) / max(1, rs_.iterations),
            "chain_seconds": rs_.chain_seconds, "chain_launches": rs_.chain_launches,
            "chain_gbs": rs_.chain_bytes / rs_.chain_seconds / 1e9 if rs_.chain_seconds else None,
            "engine": rs_.persistent, "status": rs_.status_name}
    if not args.skip_variants:
        At, bt, ct = (torch.from_numpy(v).cuda() for v in (A, b, c))
        with lpgb.LP(At, bt, ct, kernel_timing=KERNEL_TIMING_STRIDE, cuda_stream=stream.cuda_stream, price_mode=1, topk=2,
                     **extra) as lpv:
            del At, bt, ct
            lpv.solve()  # warm-up
            lpv.reset()
            torch.cuda.synchronize()
            v0 = torch.cuda.Event(enable_timing=True)
            v1 = torch.cuda.Event(enable_timing=True)
            v0.record(stream)
            rv = lpv.solve()
            v1.record(stream)
            torch.cuda.synchronize()
            tv = v0.elapsed_time(v1) * 1e-3
            zv = lpv.solution()[2]
        variants["bf16_price"] = {
            "value": rv.iterations / tv, "unit": "iters/s", "time_to_optimum_s": tv,
            "pivots_per_solve": rv.iterations, "objective": zv,
            "objective_rel_err_vs_fp64_path": abs(zv - z) / max(1.0, abs(z)),
            "objective_rel_err_vs_oracle": _rel_err(zv, z_oracle),
            "us_per_price": 1e6 * rv.price_seconds / max(1, rv.price_launches),
            "price_hbm_gbs": rv.price_bytes / rv.price_seconds / 1e9 if rv.price_seconds else None,
            "screen_passes": rv.screen_passes, "full_fp64_passes": rv.full_passes,
            "status": rv.status_name}

    if not args.skip_variants:
        # variant: Case 2 out of core -- B^-1 (134 MB) in pinned host memory, streamed through
        # two 32 MB device buffers in row blocks every pivot; the first 256 pivots
        At, bt, ct = (torch.from_numpy(v).cuda() for v in (A, b, c))
        with lpgb.LP(At, bt, ct, cuda_stream=stream.cuda_stream, tableau_budget_mb=64.0, max_iters=256) as lpo:
            del At, bt, ct
            torch.cuda.synchronize()
            v0 = torch.cuda.Event(enable_timing=True)
            v1 = torch.cuda.Event(enable_timing=True)
            v0.record(stream)
            ro = lpo.solve()
            v1.record(stream)
            torch.cuda.synchronize()
            to = v0.elapsed_time(v1) * 1e-3
        variants["out_of_core"] = {
            "value": ro.iterations / to, "unit": "iters/s", "pivots": ro.iterations,
            "seconds": to, "budget_mb": 64.0, "blocks": ro.ooc_blocks, "block_rows": ro.ooc_block_rows,
            "host_device_gbs": ro.ooc_bytes / to / 1e9, "reinversions": ro.reinversions,
            "engine_reason": lpgb.ENGINE_REASONS.get(ro.engine_reason), "status": ro.status_name,
            "what": "the first 256 pivots of the timed workload with B^-1 in pinned host memory"}

    if not args.skip_variants and not args.skip_warmstart and rank == 0:
        variants["warm_start"] = run_warmstart(lpgb)

    cpu = None
    if rank == 0 and ws == 1 and not args.skip_cpu:
        cpu = cpu_baseline(A, b, c, args.cpu_iters)

    batched = None
    if not args.skip_batch:
        batched = run_batched(lpgb, args, rank == 0 and ws == 1 and not args.skip_cpu)

    launches = sum(r.kernel_launches + 1 for r in results)  # +1: the reset kernel of each step
    if rank == 0:
        line = {
            "metric": METRIC, "value": iters_all / elapsed, "unit": "iters/s", "n_gpus": ws,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * elapsed / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic",
            "config": {"workload": WORKLOAD["name"], "m": m, "n": n, "seed": WORKLOAD["seed"],
                       "A": "U[0,1) with 10% zeros", "reinvert_every": 64, "tabu_tenure": 7,
                       "step": "one full solve from the slack basis to optimality",
                       "l2": ("no flush: the inputs (A 268 MB, its slot-ordered copy 268 MB, B^-1 134 MB) exceed "
                              "L2 and every step's reset rebuilds the slot-ordered copy; within a solve the "
                              "structured engine keeps its live rows and columns on the chip by design"
                              if results[0].persistent == 2 else
                              "no flush: A (268 MB) + B^-1 (134 MB) streamed every pivot exceed L2"),
                       "engine": {2: "slack-structured persistent", 1: "dense persistent",
                                  0: "captured graphs"}[results[0].persistent],
                       "engine_reason": lpgb.ENGINE_REASONS.get(results[0].engine_reason),
                       "parallelism": f"replicas x{ws}"},
            "time_to_optimum_s": elapsed / args.steps,
            "pivots_per_solve": results[0].iterations,
            "reinversions_per_solve": results[0].reinversions,
            "refined_reinversions_per_solve": results[0].refined_reinversions,
            "refine_residual_max": max(r.refine_residual_max for r in results),
            "reinversion_parts_s": {"refinement_or_elimination": sum(r.reinvert_gj_seconds for r in results) / len(results),
                                    "slack_rows_assembly_bbar_y": sum(r.reinvert_assemble_seconds for r in results) / len(results),
                                    "total": reinv_s / len(results)},
            "objective": z,
            "objective_rel_err_vs_oracle": _rel_err(z, z_oracle),
            "oracle_golden": ({"objective": golden["objective"], "pivots": golden["iterations"],
                               "reinversions": golden["reinversions"],
                               "pivots_equal": results[0].iterations == golden["iterations"],
                               "source": "tests/golden/dense_real_4096x8192.json (the oracle's full solve)"}
                              if golden else None),
            "certificate": _certificate(A, b, c, x, y),
            "us_per_pivot_excl_reinversion": 1e6 * iter_s / iters,
            "reinversion_share": reinv_s / sum(r.seconds for r in results),
            "chain_hbm_gbs_excl_reinversion": chain_bytes / iter_s / 1e9,
            "roofline": roofline,
            "cpu_baseline": cpu,
            "e2e": e2e,
            "variants": variants,
            "batched": batched,
            "gpu_launches": launches,
            "clocks": clocks,
        }
        print(json.dumps(line), flush=True)
    lp.close()
    if ws > 1:
        torch.distributed.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
