#!/usr/bin/env python3
"""Benchmark of the Zippel step (prints one JSON line on rank 0).

A step is one pass of the step's device path over one batch of synthetic
input: anchor values + node check, master polynomial, the k-blocked
synthetic-division / multi-right-hand-side solve, denominators with batch
inversion, Newton in the new variable and compaction of the new skeleton.
The probes (the black-box values) are generated once by the GPU evaluator
before the timed region and stay resident in HBM; their generation time is
reported separately.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl zr|reference]
                    [--workload batched|large|serve] [--requests R]
                    [--no-large] [--no-serve] [--serve-requests R]

The default line times the step at T = 10^4, S = 21 (`value`), and adds the
large single step at T = 2^20, S = 9 (`large_step`) and the serving mix of
512 requests (`serve`), each checked against its hidden function.

--workload serve runs the serving mix instead (R requests of hidden sparse
polynomials and rational functions, 2-8 variables, T log-uniform in
[16, 2^17]): the plain per-request form (zr_reconstruct, one request after
another) against the continuous-batching server, saturated and under Poisson
arrivals at 0.7 of the server's saturated rate.

Under torchrun every rank runs an independent replica of the step on its own
GPU (the step needs no exchange between GPUs); the time is the maximum over
ranks and `value` counts the terms of all ranks.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "Zippel-step skeleton terms/s and mulmod/s vs roofline; serve p50/p99 latency"


# the sources of the solve kernel, hashed in this order to key its ncu summary
SOLVE_SOURCES = ("zr_solve.cuh", "zr_ring.cuh")


# the sources of the transform kernels
NTT_SOURCES = ("zr_fast.cu", "zr_ntt.cuh")


def kernel_traffic(kernel, workload_name, sources):
    """DRAM bytes per launch of `kernel` from the committed ncu summary of
    this workload, or None when there is none or its sources changed since."""
    import hashlib
    path = os.path.join(ROOT, "profiles", f"{kernel}_{workload_name}.md")
    csrc = os.path.join(ROOT, "paper_2505_24256_gb300", "csrc")
    try:
        fields = dict(line.split(": ", 1) for line in open(path).read().splitlines()
                      if line.startswith(("traffic_bytes_per_launch: ", "source_sha256_prefix: ")))
        h = hashlib.sha256()
        for name in sources:
            h.update(open(os.path.join(csrc, name), "rb").read())
        cur = h.hexdigest()[:16]
        if fields.get("source_sha256_prefix", "").strip() != cur:
            return None
        return int(fields["traffic_bytes_per_launch"])
    except (OSError, KeyError, ValueError):
        return None


def solve_traffic(workload_name):
    return kernel_traffic("k_solve", workload_name, SOLVE_SOURCES)


def workload(name):
    from paper_2505_24256_gb300 import workloads as W
    return {"batched": W.batched_step_1e4, "large": W.large_step_2p20}[name]()


L2_NOTE = "flushed between timed steps (256 MB write)"


def bench_config(wl, world):
    """The `config` of the JSON line; both arms print the same dict."""
    return {"workload": wl.name, "T": wl.T, "S": wl.S, "nv": wl.nv, "prime": wl.p, "l2": L2_NOTE,
            "parallelism": f"replicas{world}"}


# Instruction counts of the solve's two sequences (csrc/zr_arith.cuh), in the
# 32-bit multiply forms of the PTX they are written in: a mac8 is 4 mad.lo +
# 4 mad.hi (+ 3 addc); a Shoup chain step (mulhi64 + two mullo64) is 9 mad.lo
# + 6 mad.hi.  mad.hi issues at 32 lanes per SM per clock on this GPU, mad.lo
# at 64 on a separate pipe (zr_measure_peaks), so mad.hi bounds both.
MAC_HI, CHAIN_HI = 4, 6
HI_LANES_PER_SM_CLK = 32


def theoretical_rates(sms, sm_mhz):
    """mad.hi-issue ceilings (per second) of the MAC and of the chain step."""
    hi = sms * HI_LANES_PER_SM_CLK * sm_mhz * 1e6
    return hi / MAC_HI, hi / CHAIN_HI


class Clocks:
    """nvidia-smi samples every 200 ms while the timed region runs."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None
        self.path = None

    def start(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.gpu}", f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        rows = []
        with open(self.path) as f:
            for line in f:
                parts = [x.strip() for x in line.split(",")]
                if len(parts) >= 9:
                    rows.append(parts)
        os.unlink(self.path)
        if not rows:
            return None
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({n for r in rows for n, v in zip(names, r[5:9]) if v.lower().startswith("active")})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(rows)}


def dist_env():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def max_over_ranks(x: float, world: int, device) -> float:
    """The maximum of x over all ranks (the slowest rank's time); x itself
    on one rank.  Every rank must call it."""
    if world <= 1:
        return float(x)
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    dist.barrier()
    return float(t.item())


def job_rate(units_per_rank: float, world: int, seconds_max: float) -> float:
    """Whole-job throughput: the units all ranks processed over the slowest
    rank's time (replicas: every rank processes the same units)."""
    return world * units_per_rank / seconds_max


def cpu_baseline_step(wl, nthreads=0):
    """The oracle's step on the full workload (probes from the oracle, untimed)."""
    import oracle
    b = oracle.zippel_probes(wl.exps, wl.coef, wl.k, wl.y, wl.cs, wl.z, wl.T, nthreads=nthreads)
    t0 = time.perf_counter()
    e, c = oracle.zippel_step(wl.skel, wl.k, wl.y, wl.cs, b, nthreads=nthreads)
    dt = time.perf_counter() - t0
    ok = e.shape == wl.exps.shape and (e == wl.exps).all() and (c == wl.coef).all()
    return dt, bool(ok), b


def cpu_single_thread_step(wl, b, nroots=256):
    """The oracle's step on one host thread, from a sample: the master
    polynomial in full, the solves of nroots evenly spaced roots, scaled to
    all T roots (every root costs the same: one synthetic division and S dot
    products of length T)."""
    import numpy as np

    import oracle
    v = oracle.anchor_values(wl.skel, wl.k, wl.y)
    t0 = time.perf_counter()
    m = oracle.master_poly(v)
    t_master = time.perf_counter() - t0
    roots = np.linspace(0, wl.T - 1, min(nroots, wl.T)).astype(np.int64)
    t0 = time.perf_counter()
    oracle.tvandermonde_solve_roots(v, m, b, roots, nthreads=1)
    t_roots = time.perf_counter() - t0
    return t_master + t_roots * wl.T / roots.size, roots.size


def run_reference(args):
    """The oracle timed on the host cores (the reference arm)."""
    import oracle
    world, rank, _ = dist_env()
    if rank != 0:
        return 0
    wl = workload(args.workload)
    if args.workload != "batched":
        print(json.dumps({"impl": "reference", "unavailable": "the oracle step at T=2^20 takes hours; only the "
                          "T=10^4 workload has a reference arm"}))
        return 0
    cores = oracle.default_threads()
    b = oracle.zippel_probes(wl.exps, wl.coef, wl.k, wl.y, wl.cs, wl.z, wl.T)
    for _ in range(args.warmup):
        oracle.zippel_step(wl.skel, wl.k, wl.y, wl.cs, b)
    times = []
    for _ in range(args.steps):
        t0 = time.perf_counter()
        e, c = oracle.zippel_step(wl.skel, wl.k, wl.y, wl.cs, b)
        times.append(time.perf_counter() - t0)
    total = sum(times)
    value = args.steps * wl.T / total
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": "terms/s", "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * total / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u64", "data": "synthetic",
        "config": bench_config(wl, args.gpus),
        "cpu_baseline": {"value": value, "unit": "terms/s", "cores": cores, "kind": "oracle",
                         "sample": f"full step T={wl.T} S={wl.S} per timed step (probes from the oracle, untimed)"},
        "e2e": {"value": value, "unit": "terms/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        "mulmod_per_s": (wl.S + 2.5) * wl.T ** 2 * args.steps / total,
        "check": "generator truth" if (e.shape == wl.exps.shape and (c == wl.coef).all()) else "MISMATCH",
    }
    print(json.dumps(line), flush=True)
    return 0


def reconstruction_configs(ctx, with_oracle):
    """Full reconstructions through zr_reconstruct (host arrays in, host
    arrays out): the plain 3-variable polynomial (T = 200) and the balanced
    rational function (N 5000 / D 3000 terms); wall time per call after one
    warm-up, checked against the hidden function."""
    import numpy as np
    from paper_2505_24256_gb300 import workloads as W

    out = {}
    wl = W.plain_poly_3var()
    ctx.reconstruct(wl.nv, wl.deg, wl.seed, wl.exps, wl.coef)
    reps, t0 = 20, time.perf_counter()
    for _ in range(reps):
        (e, c), _, info = ctx.reconstruct(wl.nv, wl.deg, wl.seed, wl.exps, wl.coef)
    dt = (time.perf_counter() - t0) / reps
    ok = np.array_equal(e, wl.exps) and np.array_equal(c, wl.coef)
    r = {"ms": 1e3 * dt, "reconstructions_per_s": 1.0 / dt, "terms_per_s": wl.exps.shape[0] / dt,
         "device_ms": info["device_ms"], "steps": info["steps"], "check": "generator truth" if ok else "MISMATCH"}
    if with_oracle:
        import oracle
        t0 = time.perf_counter()
        oracle.reconstruct_poly(wl.exps, wl.coef, wl.deg, seed=wl.seed)
        r["oracle_ms"] = 1e3 * (time.perf_counter() - t0)
    out[wl.name] = r
    wl = W.balanced_5var()
    args_ = (wl.nv, wl.degN, wl.seed, wl.Nexps, wl.Ncoef, wl.Dexps, wl.Dcoef)
    ctx.reconstruct(*args_, degD=wl.degD)
    reps, t0 = 3, time.perf_counter()
    for _ in range(reps):
        (Ne, Nc), (De, Dc), info = ctx.reconstruct(*args_, degD=wl.degD)
    dt = (time.perf_counter() - t0) / reps
    ok = np.array_equal(Ne, wl.Nexps) and np.array_equal(Nc, wl.Ncoef) and np.array_equal(De, wl.Dexps) and \
        np.array_equal(Dc, wl.Dcoef)
    terms = wl.Ncoef.shape[0] + wl.Dcoef.shape[0]
    out[wl.name] = {"ms": 1e3 * dt, "terms_per_s": terms / dt, "device_ms": info["device_ms"],
                    "steps": info["steps"], "redraws": info["redraws"],
                    "check": "generator truth" if ok else "MISMATCH"}
    return out


def small_steps_modes(ctx, dev, n=64, reps=20):
    """64 small uneven Zippel steps (T = 20..66, S = 11, like the plain
    3-variable reconstruction's steps) three ways, wall clock per round of
    all 64: one asynchronous call per step, one batched call, one launch of
    a captured graph."""
    import numpy as np
    import torch

    from paper_2505_24256_gb300 import workloads as W

    def d64(a):
        return torch.from_numpy(np.ascontiguousarray(a, dtype=np.uint64).view(np.int64)).to(dev)

    keep, descs, wls = [], [], []
    for i in range(n):
        wl = W.step_workload(2000 + i, 20 + (i * 7) % 47, 2, 10, 11)
        fe, fc = torch.from_numpy(wl.exps).to(dev), d64(wl.coef)
        f = ctx.poly(wl.nv, wl.exps.shape[0], fe, fc)
        y, cs, z = d64(wl.y), d64(wl.cs), d64(wl.z)
        ske = torch.from_numpy(wl.skel).to(dev)
        b = torch.empty((wl.S, wl.T), dtype=torch.int64, device=dev)
        ctx.zippel_probes(f, wl.k, y, wl.S, cs, z, wl.T, 0, b, wl.T)
        cap = wl.T * wl.S
        oe = torch.zeros((cap, wl.nv), dtype=torch.uint8, device=dev)
        oc = torch.zeros(cap, dtype=torch.int64, device=dev)
        cnt = torch.zeros(1, dtype=torch.int64, device=dev)
        keep += [fe, fc, y, cs, z, ske, b, oe, oc, cnt]
        descs.append(dict(skel=ctx.poly(wl.nv, wl.T, ske), newvar=wl.k, S=wl.S, offset=0, y=y, samples=cs, probes=b,
                          ldb=wl.T, out_exps=oe, out_coef=oc, out_cap=cap, out_count=cnt))
        wls.append(wl)

    def per_call():
        for d in descs:
            ctx.zippel_step_async(d["skel"], d["newvar"], d["y"], d["S"], d["samples"], d["probes"], d["ldb"], 0,
                                  d["out_exps"], d["out_coef"], d["out_cap"], d["out_count"])
        ctx.stream_status()

    def batched():
        ctx.zippel_step_batched(descs)

    g = ctx.step_graph(descs)

    def graph():
        g.launch()
        g.status()

    out = {"steps": n, "T": "20..66", "S": 11, "unit": "ms per round of all steps (wall clock, host + device)"}
    for name, fn in (("one_call_per_step", per_call), ("batched_call", batched), ("graph_launch", graph)):
        for _ in range(3):
            fn()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for _ in range(reps):
            fn()
        torch.cuda.synchronize()
        out[name] = 1e3 * (time.perf_counter() - t0) / reps
    ok = all(int(d["out_count"].item()) == wl.exps.shape[0] and
             np.array_equal(d["out_coef"][:wl.exps.shape[0]].cpu().numpy().view(np.uint64), wl.coef)
             for d, wl in zip(descs, wls))
    out["check"] = "generator truth" if ok else "MISMATCH"
    g.close()
    return out


def solve_roofline(T, S, solve_avg_s, peaks, workload_name):
    """Roofline entry of the O(T^2) solve kernel k_solve: its algorithmic work
    per launch (S T^2 multiply-accumulates of the dot products, T^2 chain
    steps of the synthetic division and T^2 of the denominator q_j(v_j))
    over its average launch time, against two ceilings weighted by that mix:
    the measured rates of the two instruction sequences (zr_measure_peaks,
    this run) and their mad.hi-issue bound at the maximum SM clock."""
    macs, chain_steps = S * T * T, 2 * T * T
    ops = macs + chain_steps
    achieved = ops / solve_avg_s
    peak = ops / (macs / peaks["mac_per_s"] + chain_steps / peaks["chain_per_s"])
    sms = peaks.get("sms") or 152
    mac_th, chain_th = theoretical_rates(sms, SM_MAX_MHZ)
    peak_th = ops / (macs / mac_th + chain_steps / chain_th)
    return {"bound": "alu", "achieved": achieved / 1e9, "peak": peak / 1e9, "unit": "Gop/s",
            "frac": achieved / peak, "traffic": solve_traffic(workload_name), "traffic_unit": "bytes/launch",
            "kernel": "k_solve",
            "ops": f"S*T^2 multiply-accumulates + 2*T^2 chain steps = {ops:.4g} per launch",
            "peak_basis": "measured (zr_measure_peaks on this GPU, this run): "
                          f"{peaks['mac_per_s'] / 1e9:.0f} GMAC/s, {peaks['chain_per_s'] / 1e9:.0f} G chain "
                          "steps/s, weighted by the solve's mix",
            "peak_theoretical": peak_th / 1e9, "frac_theoretical": achieved / peak_th,
            "theoretical_basis": f"mad.hi issue: {sms} SMs x {HI_LANES_PER_SM_CLK} lanes/clk x {SM_MAX_MHZ:.0f} MHz; "
                                 f"{MAC_HI} mad.hi per MAC ({mac_th / 1e9:.0f} G/s), {CHAIN_HI} per chain step "
                                 f"({chain_th / 1e9:.0f} G/s), weighted by the solve's mix"}


def quadratic_form_bench(ctx, step, flush, stream, steps, wl, peaks, oe, oc, ms_auto):
    """The step with the O(T^2) solve of Sec. 2.2 forced: one warm-up, then
    `steps` timed with the L2 flushed before each; k_solve's roofline from
    the profiler's solve phase; output against generator truth."""
    import numpy as np
    import torch
    T, S = wl.T, wl.S
    ctx.solve_method(ctx.SOLVE_QUADRATIC)
    try:
        flush.zero_()
        step()
        torch.cuda.synchronize()
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
        n = 0
        for i in range(steps):
            flush.zero_()
            evs[i][0].record(stream)
            n = step()
            evs[i][1].record(stream)
        torch.cuda.synchronize()
        # phases (and k_solve's launch time) from a second, profiled pass
        ctx.profile(True)
        for i in range(steps):
            flush.zero_()
            step()
        torch.cuda.synchronize()
        solve_ms, solve_n = ctx.profile_query("solve")
        phases = {ph: ctx.profile_query(ph)[0] / max(steps, 1) for ph in ctx.PHASES[:7]}
        ctx.profile(False)
    finally:
        ctx.solve_method(ctx.SOLVE_AUTO)
    ms = sum(a.elapsed_time(b) for a, b in evs) / steps
    ok = n == wl.exps.shape[0] and np.array_equal(oe[:n].cpu().numpy(), wl.exps) and \
        np.array_equal(oc[:n].cpu().numpy().view(np.uint64), wl.coef)
    return {"ms_per_step": ms, "terms_per_s": T / (ms / 1e3), "mulmod_per_s": (S + 2.5) * T * T / (ms / 1e3),
            "fast_speedup": ms / ms_auto, "steps": steps,
            "what": "the same step with the O(T^2) solve of Sec. 2.2 (k_solve) forced",
            "roofline": solve_roofline(T, S, solve_ms / max(solve_n, 1) / 1e3, peaks, wl.name),
            "phase_ms": phases, "check": "generator truth" if ok else "MISMATCH"}


def evaluator_method(ctx, call):
    """Which evaluator the library takes for a probe call: "transposed tree"
    when the call launched the transform kernels, else "matrix-vector"."""
    import torch
    torch.cuda.synchronize()
    ctx.profile(True)
    call()
    torch.cuda.synchronize()
    n = ctx.profile_query("ntt")[1]
    ctx.profile(False)
    return "transposed tree" if n else "matrix-vector"


def probe_gen_entry(ms, S, T, G, peaks, method):
    """The probe evaluator's figure: S x T probes of a function whose G terms
    have distinct anchor monomials.  The matrix-vector evaluator does S T G
    multiply-accumulates (rated against the measured MAC peak); the
    transposed subproduct tree computes the same values with O((G + S T)
    log^2) transform work, so only its time is given."""
    e = {"ms": ms, "evaluator": method, "probes": S * T, "terms": G}
    if method == "matrix-vector":
        macs = S * T * G
        e.update({"macs": macs, "mac_per_s": macs / (ms * 1e-3),
                  "frac_of_measured_mac_peak": macs / (ms * 1e-3) / peaks["mac_per_s"]})
    else:
        e["probes_per_s"] = S * T / (ms * 1e-3)
    return e


# the profiler phases timing the fast path's transform kernels, their kernels
FAST_KERNELS = (("desc", "k_desc_cluster"), ("ntt", "k_desc_tile, k_ntt_local"), ("psum", "k_power_sums"))


def fast_roofline(ctx, peaks, workload_name, steps, step_ms):
    """Roofline entry of the O(T log^2 T) solve's dominant kernel: of the
    descent's cluster level kernel k_desc_cluster, the transform tile kernels
    k_desc_tile and k_ntt_local and the direct power sums kernel k_power_sums, the one with the
    largest time in the profiled steps (each launch timed alone).  Its work
    per launch (radix-2 butterflies, n/2 per stage of each transform it runs,
    or the power sums' T^2 Shoup steps, counted by the library's profiler)
    over its average launch time (CUDA events around each launch on the
    launching stream, this run), against the measured rate of the same
    operation with its operands in registers (zr_measure_peaks, this run):
    the butterfly, or the Shoup chain step.  The other kernels' figures are
    given beside it."""
    entries = []
    for phase, kernel in FAST_KERNELS:
        ms, n = ctx.profile_query(phase)
        work = ctx.profile_work(phase)
        if n <= 0 or ms <= 0:
            continue
        achieved = work / (ms * 1e-3)
        if phase == "psum":
            peak = peaks["chain_per_s"]
            ops = (f"Shoup steps v_j^k -> v_j^(k+1), T^2 per launch: {work / n:.4g} per launch on average, "
                   f"{n / max(steps, 1):.0f} launches per step")
            basis = ("measured (zr_measure_peaks on this GPU, this run): Shoup chain steps (mulhi64 + two "
                     f"mullo64), operands in registers, {peak / 1e9:.0f} G/s")
        else:
            peak = peaks["butterfly_per_s"]
            ops = (f"radix-2 butterflies, n/2 per stage of each transform: {work / n:.4g} per launch on average, "
                   f"{n / max(steps, 1):.0f} launches per step")
            basis = ("measured (zr_measure_peaks on this GPU, this run): forward butterflies on 32-bit "
                     f"residues with a Shoup twiddle, operands in registers, {peak / 1e9:.0f} G/s")
        entries.append((ms, {
            "bound": "alu", "achieved": achieved / 1e9, "peak": peak / 1e9, "unit": "Gop/s",
            "frac": achieved / peak,
            "traffic": kernel_traffic(kernel.split(",")[0], workload_name, NTT_SOURCES),
            "traffic_unit": "bytes/launch", "kernel": kernel, "ops": ops,
            "launch_ms": ms / n, "share_of_step": ms / max(steps, 1) / step_ms,
            "peak_basis": basis}))
    if not entries:
        return None
    entries.sort(key=lambda x: -x[0])
    main = dict(entries[0][1])
    if len(entries) > 1:
        main["next_kernel"] = entries[1][1]
    if len(entries) > 2:
        main["third_kernel"] = entries[2][1]
    return main


SM_MAX_MHZ = 2070.0   # GB300 maximum SM clock (the clocks record of each run gives the live value)


def run_zr(args):
    import numpy as np
    import torch
    import torch.distributed as dist

    import __graft_entry__ as ge
    from paper_2505_24256_gb300 import zr

    world, rank, local = dist_env()
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device(f"cuda:{local}"))
    torch.cuda.set_device(local)
    dev = torch.device(f"cuda:{local}")
    ge.build()
    wl = workload(args.workload)
    T, S, nv, k = wl.T, wl.S, wl.nv, wl.k

    def d64(a):
        return torch.from_numpy(np.ascontiguousarray(a, dtype=np.uint64).view(np.int64)).to(dev)

    ctx = zr.Context(wl.p)
    stream = torch.cuda.current_stream()
    # resident inputs: hidden function (for the evaluator), skeleton, anchor, samples, rest values
    fe, fc = torch.from_numpy(wl.exps).to(dev), d64(wl.coef)
    f = ctx.poly(nv, wl.exps.shape[0], fe, fc)
    y, cs, z = d64(wl.y), d64(wl.cs), d64(wl.z)
    ske = torch.from_numpy(wl.skel).to(dev)
    skel = ctx.poly(nv, T, ske)
    b = torch.empty((S, T), dtype=torch.int64, device=dev)
    # probes by the GPU evaluator (outside the timed step): the first call,
    # then, when that is short, the median of three more
    probe_times = []
    for _ in range(4):
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        ctx.zippel_probes(f, k, y, S, cs, z, T, 0, b, T)
        e1.record(stream)
        torch.cuda.synchronize()
        probe_times.append(e0.elapsed_time(e1))
        if probe_times[0] > 100.0:
            break
    probe_ms = probe_times[0] if len(probe_times) == 1 else sorted(probe_times[1:])[1]
    probe_method = evaluator_method(ctx, lambda: ctx.zippel_probes(f, k, y, S, cs, z, T, 0, b, T))
    cap = T * S
    oe = torch.zeros((cap, nv), dtype=torch.uint8, device=dev)
    oc = torch.zeros(cap, dtype=torch.int64, device=dev)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.int32, device=dev)   # 256 MB > L2 (129 MB)

    def step():
        return ctx.zippel_step(skel, k, y, S, cs, b, T, 0, oe, oc, cap)

    # launch plan: autotuned for this shape when tuning is affordable, else the model
    if S * T * T <= 10**11:
        ctx.autotune_step(T, S, 24)
    plan = ctx.step_plan(T, S)
    # measured ceilings of the solve's two instruction sequences (MAC, chain step)
    peaks = ctx.measure_peaks()

    for _ in range(args.warmup):
        flush.zero_()
        step()
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    clocks = Clocks(local)
    clocks.start()
    launches0 = zr.launch_count()
    total_ms = 0.0
    n = 0
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    for i in range(args.steps):
        flush.zero_()                      # L2 flushed between timed steps (outside the events)
        evs[i][0].record(stream)
        n = step()
        evs[i][1].record(stream)
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    launches = zr.launch_count() - launches0
    clk = clocks.stop()
    step_times = sorted(a.elapsed_time(bb) for a, bb in evs)
    total_ms = sum(step_times)
    median_ms = step_times[len(step_times) // 2] if len(step_times) % 2 else \
        0.5 * (step_times[len(step_times) // 2 - 1] + step_times[len(step_times) // 2])
    # the same steps again with the library's profiler on (CUDA events around
    # the phases and around each transform launch): phase times and the
    # dominant kernel's launch times, outside the timed region above
    ctx.profile(True)
    pevs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    for i in range(args.steps):
        flush.zero_()
        pevs[i][0].record(stream)
        step()
        pevs[i][1].record(stream)
    torch.cuda.synchronize()
    prof_step_ms = sum(a.elapsed_time(bb) for a, bb in pevs) / args.steps
    solve_ms, solve_n = ctx.profile_query("solve")
    fast_n = ctx.profile_query("fast")[1]
    phases = {ph: ctx.profile_query(ph)[0] / max(args.steps, 1) for ph in zr.Context.PHASES[:7] + ("fast", "ntt", "desc")}
    ntt_roof = fast_roofline(ctx, peaks, wl.name, args.steps, prof_step_ms) if fast_n else None
    ctx.profile(False)
    total_ms = max_over_ranks(total_ms, world, dev)
    # the output of the last timed step against generator truth
    ok = n == wl.exps.shape[0] and np.array_equal(oe[:n].cpu().numpy(), wl.exps) and \
        np.array_equal(oc[:n].cpu().numpy().view(np.uint64), wl.coef)
    # when the library chose the O(T log^2 T) solve: the same step with the
    # paper's O(T^2) solve (k_solve), timed the same way, with its roofline
    quad = quadratic_form_bench(ctx, step, flush, stream, args.steps, wl, peaks, oe, oc, total_ms / args.steps) \
        if fast_n else None

    # end to end through the C ABI with host buffers (pinned), copies inside the timed region
    h_exps = torch.from_numpy(wl.skel).pin_memory()
    h_y = torch.from_numpy(wl.y.view(np.int64)).pin_memory()
    h_cs = torch.from_numpy(wl.cs.view(np.int64)).pin_memory()
    h_b = b.cpu().pin_memory()
    h_oe = torch.zeros((cap, nv), dtype=torch.uint8).pin_memory()
    h_oc = torch.zeros(cap, dtype=torch.int64).pin_memory()
    hskel = ctx.poly(nv, T, h_exps)
    e2e_steps = max(1, min(args.steps, 10))
    ctx.zippel_step_host(hskel, k, h_y, S, h_cs, h_b, T, 0, h_oe, h_oc, cap)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(e2e_steps):
        ne = ctx.zippel_step_host(hskel, k, h_y, S, h_cs, h_b, T, 0, h_oe, h_oc, cap)
    e2e_s = (time.perf_counter() - t0) / e2e_steps
    e2e_ok = ne == wl.exps.shape[0] and np.array_equal(h_oc[:ne].numpy().view(np.uint64), wl.coef)
    e2e_s = max_over_ranks(e2e_s, world, dev)

    # the plain form on the same GPU: one single-right-hand-side system per
    # launch sequence (S of them), then Newton; probes and nodes as above
    v = torch.empty(T, dtype=torch.int64, device=dev)
    cpl = torch.empty((S, T), dtype=torch.int64, device=dev)
    gpl = torch.empty((S, T), dtype=torch.int64, device=dev)
    systems = [dict(T=T, S=1, v=v, b=b[s], ldb=T, c=cpl[s], ldc=T) for s in range(S)]

    def plain_step():
        ctx.anchor_values(T, nv, ske, k, y, 0, v)
        ctx.solve_method(ctx.SOLVE_QUADRATIC)      # the paper's O(T^2) solve, one system per launch sequence
        ctx.vandermonde_solve(systems, plain=True)
        ctx.solve_method(ctx.SOLVE_AUTO)
        ctx.newton_batched(T, S, cs, cpl, T, gpl)

    plain_reps = max(1, min(args.steps, 5))
    plain_step()
    torch.cuda.synchronize()
    pevs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(plain_reps)]
    for i in range(plain_reps):
        flush.zero_()
        pevs[i][0].record(stream)
        plain_step()
        pevs[i][1].record(stream)
    torch.cuda.synchronize()
    plain_ms = sum(a.elapsed_time(bb) for a, bb in pevs) / plain_reps
    plain_ok = np.array_equal(gpl.cpu().numpy().view(np.uint64).T.reshape(-1), wl.coef)

    # the same step as a captured graph (one launch per step)
    graph = ctx.step_graph([dict(skel=skel, newvar=k, S=S, offset=0, y=y, samples=cs, probes=b, ldb=T, out_exps=oe,
                                 out_coef=oc, out_cap=cap, out_count=torch.zeros(1, dtype=torch.int64, device=dev))])
    gevs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(plain_reps)]
    for i in range(plain_reps):
        flush.zero_()
        gevs[i][0].record(stream)
        graph.launch()
        gevs[i][1].record(stream)
    graph.status()
    graph_ms = sum(a.elapsed_time(bb) for a, bb in gevs) / plain_reps
    graph_kernels = graph.kernels
    graph.close()
    small = small_steps_modes(ctx, dev)
    recons = reconstruction_configs(ctx, with_oracle=world == 1 and not args.no_cpu_baseline) \
        if args.workload == "batched" else None
    # the largest single-GPU configuration (T = 2^20) and the serving mix, on
    # every rank (replicas), in the same line
    large = None
    if args.workload == "batched" and not args.no_large:
        large = large_step_bench(ctx, dev, flush, peaks, steps=2, warmup=1)
    serve = None
    if args.workload == "batched" and not args.no_serve:
        serve = serve_mix(args, args.serve_requests, 1005 + 1000 * rank)

    if rank != 0:
        ctx.close()
        if world > 1:
            dist.destroy_process_group()
        return 0

    solve_avg_s = solve_ms / max(solve_n, 1) / 1e3
    ms_per_step = total_ms / args.steps
    W = (S + 2.5) * T * T
    line = {
        "metric": METRIC,
        "value": job_rate(T * args.steps, world, total_ms / 1e3),
        "unit": "terms/s",
        "n_gpus": world, "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_per_step,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u64", "data": "synthetic",
        "config": bench_config(wl, world),
        "solve": "O(T log^2 T) (subproduct tree, transforms over five 30-bit primes)" if fast_n
                 else "O(T^2) (Sec. 2.2, k_solve)",
        # mulmod/s of the O(T^2) form: S T^2 multiply-accumulates + 2.5 T^2 chain and denominator steps per step
        "mulmod_per_s": quad["mulmod_per_s"] * world if quad else world * W * args.steps / (total_ms / 1e3),
        # the median step of this rank (the per-step figure the paper reports)
        "median": {"ms_per_step": median_ms, "terms_per_s": T / (median_ms / 1e3), "steps": len(step_times)},
        "roofline": ntt_roof if fast_n else solve_roofline(T, S, solve_avg_s, peaks, wl.name),
        "quadratic_form": quad,
        "peaks_measured": {"mac_per_s": peaks["mac_per_s"], "chain_per_s": peaks["chain_per_s"],
                           "imad_lo_per_s": peaks["imad_lo_per_s"], "imad_hi_per_s": peaks["imad_hi_per_s"],
                           "butterfly_per_s": peaks["butterfly_per_s"]},
        "plain_form": {"ms_per_step": plain_ms, "terms_per_s": world * T / (plain_ms / 1e3),
                       "batched_speedup": plain_ms / ms_per_step,
                       "what": f"{S} single-RHS systems, one launch sequence each, + Newton",
                       "check": "generator truth" if plain_ok else "MISMATCH"},
        "graph": {"ms_per_step": graph_ms, "kernels_per_launch": graph_kernels},
        "small_steps": small,
        "reconstructions": recons,
        "large_step": large,
        "serve": serve,
        "phase_ms": phases,
        "plan": {"s_tile": plan[0], "k_blocks": plan[1]},
        "probe_gen_ms": probe_ms,
        "probe_gen": probe_gen_entry(probe_ms, S, T, T, peaks, probe_method),
        "e2e": {"value": job_rate(T, world, e2e_s), "unit": "terms/s",
                "h2d_bytes_per_step": T * nv + 8 * k + 8 * S + 8 * S * T,
                "d2h_bytes_per_step": min(cap, T * S) * (nv + 8) + 12},
        "gpu_launches": int(launches),
        "clocks": clk,
        "check": "generator truth" if (ok and e2e_ok and (large is None or large["check"] == "generator truth")
                                       and (serve is None or serve["check"] == "generator truth")) else "MISMATCH",
    }
    if world == 1 and not args.no_cpu_baseline and args.workload == "batched":
        import oracle
        cores = oracle.default_threads()
        dt, cok, ob = cpu_baseline_step(wl)
        st, nr = cpu_single_thread_step(wl, ob)
        line["cpu_baseline"] = {"value": T / dt, "unit": "terms/s", "cores": cores, "kind": "oracle",
                                "sample": f"one full step T={T} S={S} (probes from the oracle, untimed)",
                                "check": "generator truth" if cok else "MISMATCH",
                                "single_thread": {"value": T / st, "unit": "terms/s", "cores": 1,
                                                  "sample": f"master polynomial in full + {nr} of the {T} roots' "
                                                            "solves, scaled to all roots"}}
    print(json.dumps(line), flush=True)
    ctx.close()
    if world > 1:
        dist.destroy_process_group()
    return 0


def large_step_bench(ctx, dev, flush, peaks, steps, warmup):
    """The large single step, T = 2^20 terms in 7 variables, S = 9: probes by
    the GPU evaluator (timed apart), then `warmup` untimed and `steps` timed
    steps with the L2 flushed before each, checked against the hidden function;
    the plain one-system-per-launch form is timed on one of its S identical
    single-right-hand-side systems and scaled by S."""
    import numpy as np
    import torch

    from paper_2505_24256_gb300 import workloads as W

    def d64(a):
        return torch.from_numpy(np.ascontiguousarray(a, dtype=np.uint64).view(np.int64)).to(dev)

    wl = W.large_step_2p20()
    T, S, nv, k = wl.T, wl.S, wl.nv, wl.k
    ctx.solve_method(ctx.SOLVE_AUTO)
    stream = torch.cuda.current_stream()
    fe, fc = torch.from_numpy(wl.exps).to(dev), d64(wl.coef)
    f = ctx.poly(nv, wl.exps.shape[0], fe, fc)
    y, cs, z = d64(wl.y), d64(wl.cs), d64(wl.z)
    ske = torch.from_numpy(wl.skel).to(dev)
    skel = ctx.poly(nv, T, ske)
    b = torch.empty((S, T), dtype=torch.int64, device=dev)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    ctx.zippel_probes(f, k, y, S, cs, z, T, 0, b, T)
    e1.record(stream)
    torch.cuda.synchronize()
    probe_ms = e0.elapsed_time(e1)
    probe_method = evaluator_method(ctx, lambda: ctx.zippel_probes(f, k, y, S, cs, z, T, 0, b, T))
    del fe, fc
    cap = T * S
    oe = torch.zeros((cap, nv), dtype=torch.uint8, device=dev)
    oc = torch.zeros(cap, dtype=torch.int64, device=dev)
    for _ in range(warmup):
        flush.zero_()
        ctx.zippel_step(skel, k, y, S, cs, b, T, 0, oe, oc, cap)
    torch.cuda.synchronize()
    clocks = Clocks(torch.cuda.current_device())
    clocks.start()
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
    n = 0
    for i in range(steps):
        flush.zero_()
        evs[i][0].record(stream)
        n = ctx.zippel_step(skel, k, y, S, cs, b, T, 0, oe, oc, cap)
        evs[i][1].record(stream)
    torch.cuda.synchronize()
    clk = clocks.stop()
    times = [a.elapsed_time(bb) for a, bb in evs]
    # phases and the dominant kernel's launches from a second, profiled pass
    ctx.profile(True)
    pevs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
    for i in range(steps):
        flush.zero_()
        pevs[i][0].record(stream)
        ctx.zippel_step(skel, k, y, S, cs, b, T, 0, oe, oc, cap)
        pevs[i][1].record(stream)
    torch.cuda.synchronize()
    prof_ms = sum(a.elapsed_time(bb) for a, bb in pevs) / steps
    fast_ms, fast_n = ctx.profile_query("fast")
    phases = {ph: ctx.profile_query(ph)[0] / max(steps, 1) for ph in ctx.PHASES[:7] + ("fast", "ntt", "desc")}
    fast_roof = fast_roofline(ctx, peaks, wl.name, steps, prof_ms)
    ctx.profile(False)
    ok = n == wl.exps.shape[0] and np.array_equal(oe[:n].cpu().numpy(), wl.exps) and \
        np.array_equal(oc[:n].cpu().numpy().view(np.uint64), wl.coef)
    ms = sum(times) / len(times)
    # the same step with the paper's O(T^2) solve (k_solve): one warm-up, one timed
    ctx.solve_method(ctx.SOLVE_QUADRATIC)
    flush.zero_()
    ctx.zippel_step(skel, k, y, S, cs, b, T, 0, oe, oc, cap)
    ctx.profile(True)
    flush.zero_()
    torch.cuda.synchronize()
    e0.record(stream)
    nq = ctx.zippel_step(skel, k, y, S, cs, b, T, 0, oe, oc, cap)
    e1.record(stream)
    torch.cuda.synchronize()
    quad_ms = e0.elapsed_time(e1)
    solve_ms, solve_n = ctx.profile_query("solve")
    qphases = {ph: ctx.profile_query(ph)[0] for ph in ctx.PHASES[:7]}
    ctx.profile(False)
    ctx.solve_method(ctx.SOLVE_AUTO)
    qok = nq == wl.exps.shape[0] and np.array_equal(oc[:nq].cpu().numpy().view(np.uint64), wl.coef)
    del oe, oc
    # the plain form: one single-right-hand-side system per launch sequence;
    # its S systems are identical in cost, so one is timed and scaled by S
    v = torch.empty(T, dtype=torch.int64, device=dev)
    c1 = torch.empty(T, dtype=torch.int64, device=dev)
    ctx.anchor_values(T, nv, ske, k, y, 0, v)
    flush.zero_()
    torch.cuda.synchronize()
    e0.record(stream)
    ctx.solve_method(ctx.SOLVE_QUADRATIC)
    ctx.vandermonde_solve([dict(T=T, S=1, v=v, b=b[0], ldb=T, c=c1, ldc=T)], plain=True)
    ctx.solve_method(ctx.SOLVE_AUTO)
    e1.record(stream)
    torch.cuda.synchronize()
    plain_one_ms = e0.elapsed_time(e1)
    # the first system's solution is c_j = g_j(c_0) = sum_e G[j, e] c_0^e:
    # 64 sampled roots against the hidden coefficients (Python integers)
    plain_ok = True
    idx = np.linspace(0, T - 1, 64).astype(np.int64)
    got = c1.cpu().numpy().view(np.uint64)[idx]
    c0 = int(wl.cs[0])
    for jj, gv in zip(idx, got):
        want = 0
        for e in range(S - 1, -1, -1):
            want = (want * c0 + int(wl.G[jj, e])) % wl.p
        plain_ok &= int(gv) == want
    W_ = (S + 2.5) * T * T
    return {
        "workload": wl.name, "T": T, "S": S, "nv": nv, "steps": steps, "warmup": warmup,
        "solve": "O(T log^2 T) (subproduct tree, transforms over five 30-bit primes)",
        "ms_per_step": ms, "terms_per_s": T / (ms / 1e3),
        "fast_solve_ms": fast_ms / max(fast_n, 1),
        "fast_solve_note": "from the profiled pass (the whole solve then runs on the call's stream)",
        "roofline": fast_roof,
        "phase_ms": phases,
        "quadratic_form": {"ms_per_step": quad_ms, "terms_per_s": T / (quad_ms / 1e3),
                           "mulmod_per_s": W_ / (quad_ms / 1e3), "fast_speedup": quad_ms / ms,
                           "what": "the same step with the O(T^2) solve of Sec. 2.2 (k_solve); one warm-up, one timed",
                           "roofline": solve_roofline(T, S, solve_ms / max(solve_n, 1) / 1e3, peaks, wl.name),
                           "phase_ms": qphases,
                           "check": "generator truth" if qok else "MISMATCH"},
        "plain_form": {"ms_per_step": plain_one_ms * S, "terms_per_s": T / (plain_one_ms * S / 1e3),
                       "batched_speedup": plain_one_ms * S / ms,
                       "quadratic_batched_speedup": plain_one_ms * S / quad_ms,
                       "what": f"{S} single-RHS systems, one launch sequence each; one timed "
                               f"({plain_one_ms:.0f} ms) and scaled by {S} (identical cost)",
                       "check": "generator truth (64 sampled roots)" if plain_ok else "MISMATCH"},
        "probe_gen": probe_gen_entry(probe_ms, S, T, T, peaks, probe_method),
        "clocks": clk,
        "l2": "flushed before each timed step (256 MB write); the step's inputs exceed L2",
        "check": "generator truth" if (ok and qok and plain_ok) else "MISMATCH",
    }


def serve_stats(lat_ms):
    import numpy as np
    a = np.sort(np.asarray(lat_ms, dtype=np.float64))
    q = lambda f: float(a[min(len(a) - 1, int(f * (len(a) - 1) + 0.5))])
    return {"p50_ms": q(0.5), "p99_ms": q(0.99), "mean_ms": float(a.mean())}


def serve_mix(args, nreq, seed):
    """The serving mix of nreq requests (hidden sparse polynomials and rational
    functions, 2-8 variables, T log-uniform in [16, tmax]):
      * the plain per-request form, zr_reconstruct once per request, back to
        back (throughput and service times);
      * the continuous-batching server with every request submitted at once
        (saturated throughput);
      * the server under Poisson arrivals at 0.7 of its saturated rate;
      * the plain form under the same arrivals, run in real time (a request
        starts at its arrival or when the previous one ends).
    Every result is checked against its hidden function."""
    import numpy as np
    import torch

    from paper_2505_24256_gb300 import workloads as W
    from paper_2505_24256_gb300 import zr

    reqs = W.serve_requests(nreq, seed=seed, tmax=args.tmax)
    wls = [W.serve_blackbox(r) for r in reqs]
    reqobjs = []
    for wl in wls:
        if isinstance(wl, W.RationalWorkload):
            reqobjs.append(zr.make_request(wl.nv, wl.degN, wl.seed, wl.Nexps, wl.Ncoef, wl.Dexps, wl.Dcoef,
                                           degD=wl.degD))
        else:
            reqobjs.append(zr.make_request(wl.nv, wl.deg, wl.seed, wl.exps, wl.coef))
    terms = sum(int(wl.Ncoef.shape[0] + wl.Dcoef.shape[0]) if isinstance(wl, W.RationalWorkload)
                else int(wl.coef.shape[0]) for wl in wls)

    def truth(wl, res):
        (e, c), D, _ = res
        if isinstance(wl, W.RationalWorkload):
            return np.array_equal(e, wl.Nexps) and np.array_equal(c, wl.Ncoef) and D is not None and \
                np.array_equal(D[0], wl.Dexps) and np.array_equal(D[1], wl.Dcoef)
        return np.array_equal(e, wl.exps) and np.array_equal(c, wl.coef)

    def plain_one(ctx, wl):
        if isinstance(wl, W.RationalWorkload):
            return ctx.reconstruct(wl.nv, wl.degN, wl.seed, wl.Nexps, wl.Ncoef, wl.Dexps, wl.Dcoef, degD=wl.degD)
        return ctx.reconstruct(wl.nv, wl.deg, wl.seed, wl.exps, wl.coef)

    ctx = zr.Context(W.P63)
    for wl in wls[:min(args.warmup, len(wls))]:
        plain_one(ctx, wl)
    torch.cuda.synchronize()
    clocks = Clocks(torch.cuda.current_device())
    clocks.start()
    launches0 = zr.launch_count()
    # (1) plain per-request form, back to back
    svc = []
    ok_plain = True
    t_plain0 = time.perf_counter()
    for wl in wls:
        t0 = time.perf_counter()
        res = plain_one(ctx, wl)
        svc.append(time.perf_counter() - t0)
        ok_plain &= truth(wl, res)
    plain_s = time.perf_counter() - t_plain0

    def serve(gaps):
        c = zr.Context(W.P63)
        srv = zr.Server(c, args.serve_budget_gb << 30, args.slots)
        arrivals = []
        tickets = []
        t0 = time.perf_counter()
        for (req, _keep), g in zip(reqobjs, gaps):
            if g > 0:
                target = (arrivals[-1] if arrivals else 0.0) + g
                while time.perf_counter() - t0 < target:
                    time.sleep(min(0.0005, max(0.0, target - (time.perf_counter() - t0))))
            arrivals.append(time.perf_counter() - t0)
            tickets.append(srv.submit(req))
        outs = [srv.wait(t, timeout_s=900) for t in tickets]
        st = srv.stats()
        srv.close()
        c.close()
        ok = all(truth(wl, r) for wl, r in zip(wls, outs))
        return st, ok, outs

    # (2) saturated: everything submitted at once -> server capacity
    sat, ok_sat, _ = serve([0.0] * len(wls))
    cap_rps = sat["completed"] / sat["wall_s"]
    # (3) Poisson arrivals at 0.7 x the saturated rate
    lam = 0.7 * cap_rps
    rng = np.random.default_rng(seed)
    gaps = list(rng.exponential(1.0 / lam, size=len(wls)))
    poi, ok_poi, outs = serve(gaps)
    # (4) the plain form under the same arrivals, in real time
    arr = np.cumsum(gaps)
    lat = []
    ok_plain_poi = True
    t0 = time.perf_counter()
    for a, wl in zip(arr, wls):
        while time.perf_counter() - t0 < a:
            time.sleep(min(0.0005, max(0.0, a - (time.perf_counter() - t0))))
        res = plain_one(ctx, wl)
        lat.append(1e3 * (time.perf_counter() - t0 - a))
        ok_plain_poi &= truth(wl, res)
    plain_poi_s = time.perf_counter() - t0
    ctx.close()
    launches = zr.launch_count() - launches0
    clk = clocks.stop()
    return {
        "requests": len(wls), "seed": seed, "tmax": args.tmax, "terms": terms, "slots": args.slots,
        "mem_budget_gb": args.serve_budget_gb,
        "serve_saturated": {"terms_per_s": sat["terms_per_s"], "requests_per_s": cap_rps, "p50_ms": sat["p50_ms"],
                            "p99_ms": sat["p99_ms"], "wall_s": sat["wall_s"], "ticks": sat["ticks"],
                            "batch_entries": sat["batch_entries"], "max_active": sat["max_active"]},
        "serve_poisson": {"lambda_per_s": lam, "terms_per_s": poi["terms_per_s"], "p50_ms": poi["p50_ms"],
                          "p99_ms": poi["p99_ms"], "mean_ms": poi["mean_ms"], "max_active": poi["max_active"]},
        "plain_per_request": {"terms_per_s": terms / plain_s, "requests_per_s": len(wls) / plain_s,
                              "service_ms": serve_stats([1e3 * x for x in svc]),
                              "poisson_same_arrivals": dict(serve_stats(lat), wall_s=plain_poi_s,
                                                            how="measured: run in real time under the same "
                                                                "arrivals, one request at a time")},
        "saturated_speedup": sat["terms_per_s"] / (terms / plain_s),
        "gpu_launches": int(launches),
        "clocks": clk,
        "h2d_bytes_per_request": int(sum(o[0].bb.TN * (o[0].bb.nv + 8) + o[0].bb.TD * (o[0].bb.nv + 8)
                                         for o in reqobjs) / max(1, len(wls))),
        "d2h_bytes_per_request": int(sum((r[0][1].shape[0] + (0 if r[1] is None else r[1][1].shape[0]))
                                         * (r[0][0].shape[1] + 8) for r in outs) / max(1, len(wls))),
        "check": "generator truth" if (ok_plain and ok_sat and ok_poi and ok_plain_poi) else "MISMATCH",
    }


def run_serve(args):
    """The serving mix alone (--workload serve), its own JSON line."""
    import torch

    import __graft_entry__ as ge

    world, rank, local = dist_env()
    torch.cuda.set_device(local)
    ge.build()
    r = serve_mix(args, args.requests, 1005 + 1000 * rank)
    sat = r["serve_saturated"]
    line = {
        "metric": METRIC,
        "value": sat["terms_per_s"], "unit": "terms/s",
        "n_gpus": world, "steps": r["requests"], "warmup": args.warmup,
        "ms_per_step": 1e3 * sat["wall_s"] / max(1, r["requests"]),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u64", "data": "synthetic",
        "config": {"workload": f"serve_{r['requests']}_requests", "requests": r["requests"], "seed": 1005,
                   "tmax": args.tmax, "terms": r["terms"], "slots": args.slots,
                   "mem_budget_gb": args.serve_budget_gb,
                   "l2": "inputs of the larger requests exceed L2", "parallelism": f"replicas{world}"},
        "e2e": {"value": sat["terms_per_s"], "unit": "terms/s", "h2d_bytes_per_step": r["h2d_bytes_per_request"],
                "d2h_bytes_per_step": r["d2h_bytes_per_request"]},
        "gpu_launches": r["gpu_launches"],
        "clocks": r["clocks"],
        "serve": r,
        "check": r["check"],
    }
    if rank == 0:
        print(json.dumps(line), flush=True)
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="zr", choices=["zr", "reference"])
    ap.add_argument("--workload", default="batched", choices=["batched", "large", "serve"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--requests", type=int, default=512, help="serving mix size (--workload serve)")
    ap.add_argument("--serve-requests", type=int, default=512, help="serving mix size in the default line")
    ap.add_argument("--no-large", action="store_true", help="leave the T = 2^20 step out of the default line")
    ap.add_argument("--no-serve", action="store_true", help="leave the serving mix out of the default line")
    ap.add_argument("--tmax", type=int, default=1 << 17, help="largest request T (--workload serve)")
    ap.add_argument("--slots", type=int, default=64, help="server slots (--workload serve)")
    ap.add_argument("--serve-budget-gb", type=int, default=64, help="server memory budget (--workload serve)")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        return run_reference(args)
    if args.workload == "serve":
        return run_serve(args)
    return run_zr(args)


if __name__ == "__main__":
    rc = main()
    sys.stdout.flush()
    sys.stderr.flush()
    # Under the profiler, process-exit destructors of the CUDA libraries have
    # crashed after the result line was out: the profiling commands set
    # ZR_BENCH_HARD_EXIT=1 to leave without interpreter teardown.
    if os.environ.get("ZR_BENCH_HARD_EXIT") == "1":
        os._exit(rc or 0)
    sys.exit(rc or 0)
