"""Benchmark: multi-agent QP solves/sec at residual 1e-4, batched GPU vs plain GPU.

Workload (one step): the 4096-scenario mixed batch (N ~ U{2..32} agents,
T ~ U{20..40} steps, 2D double integrator, d_min 0.4, rho 1, |u| <= 1), FP64,
solved from scratch by ADMM to primal and dual residual 1e-4 or 500 iterations
in one persistent, graph-captured launch.  A solve is a scenario that reaches
the tolerance; scenarios stopped by the iteration cap are reported, not counted.

value      converged solves / second, inputs resident in HBM, device-timed (CUDA
           events on the launch stream around each step, L2 flushed between steps).
pipelined  the same steps device-timed over two handles on two streams taking
           alternate steps, so that one batch's tail (the last scenario groups of
           the work queue) overlaps the next batch's start.
e2e        the same metric through the C ABI from pinned host buffers: upload of
           every input array, solve, download of X, U, theta, W, status, iters,
           residuals, all inside the timed region, every step; two handles on
           two streams take alternate steps, so one step's upload and solve
           overlap the previous step's read-back.
roofline   FP64 pipe (ALU-bound): the FP64 flops that the step cannot do without, from
           the kernel's own event counters (pair-steps, EQP stages, factorized stages)
           and the share of pair-steps that are projected, over the device time, against the FP64 FMA throughput measured in the same run
           by the library's probe kernel (tadmm_fma_probe); the derived figure
           152 SMs x 4 FP64 flop/clk x 2.07 GHz = 1.259 TFLOP/s is reported beside
           it.  DRAM traffic and executed FP64 instruction counts come from the
           committed ncu summary of this kernel, used only while the kernel
           sources hash to the value recorded there.
plain_gpu  the same kernels, one scenario at a time, one launch per phase and a
           host read of the residuals every iteration, on a seeded sample; the
           work-matched speedup is the ratio of scenario-iterations per second.
extras     the other synthetic workloads (2-agent crossing, 14-agent ring,
           512-agent 3D swarm, 64 x 16-agent differentiation batch), float32 and
           double-float arithmetic and the extensions, each device-timed.
cpu_baseline  the FP64 oracle on the host cores on a bounded seeded sample
           (one scenario per core, 20 ADMM iterations each), scaled to solves/s
           with the GPU run's solves per scenario-iteration.

--impl reference runs that oracle as the reference arm (rank 0 only).
Multi-GPU (torchrun): each rank solves its own batch (scenario ids offset by
rank), no collective on the data path; whole-job value = all solves / max time.
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

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "multi-agent QP solves/sec at residual 1e-4 (batched vs plain GPU); ms/solve"
UNIT = "solves/s"
PEAK_FP64_DERIVED_TFLOPS = 152 * 4 * 2.07e9 / 1e12   # 1.259
# Solves per scenario-iteration of the 4096-scenario mixed batch at tol 1e-4,
# max_iter 500: 194 solves in 1 955 163 scenario-iterations.  A property of the
# ADMM iterates on these instances (the GPU and the oracle produce the same
# iterates and iteration counts; a GPU test checks these two numbers against a
# fresh solve, so a change of the kernels or the generator cannot leave them
# stale); the reference arm uses it to express the oracle's measured
# scenario-iteration throughput in solves/s, so the ratio of the two arms is
# the ratio of their scenario-iteration throughputs.
WORKLOAD_SOLVES, WORKLOAD_SCEN_ITERS = 194, 1955163
WORKLOAD_SOLVES_PER_SCEN_ITER = WORKLOAD_SOLVES / WORKLOAD_SCEN_ITERS
# FP64 flops that a unit cannot do without: projected pair-step, EQP stage, factorized
# stage.  The double integrator's stages fall apart into one two-state, one-input
# recursion per axis: 26 flops of a pass and 35 of a factorization each (its zeros are
# not counted).  A pair-step takes FP64 (differences, product, step and its term in
# either agent's sum) only where it pushes or may push; the others end at a float32 test
# and count nothing.
FLOPS_2D = (16.0, 52.0, 70.0)       # nx = 4, nu = 2
FLOPS_3D = (23.0, 78.0, 105.0)      # nx = 6, nu = 3
# Share of the pair-steps of the 4096-scenario batch over 500 iterations that are
# projected: 4.033e8 of 1.071e10, counted once in a copy of the kernel (over the first
# 100 iterations 5.2 in a hundred).  A property of the iterates.  For other runs the
# share is not known and counts as 0, so that their flops are a lower bound.
WORKLOAD_PROJECTED_SHARE = 0.0377
FLOPS_PAIRSTEP, FLOPS_EQP_STAGE, FLOPS_FACT_STAGE = FLOPS_2D
COUNTERS_FILE = os.path.join(ROOT, "profiles", "k_batched_mixed4096_counters.txt")


def parse():
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=3)
    p.add_argument("--warmup", type=int, default=3)
    p.add_argument("--impl", default="ours", choices=["ours", "reference"])
    p.add_argument("--precision", type=int, default=64)
    p.add_argument("--n-scen", type=int, default=4096)
    p.add_argument("--tol", type=float, default=1e-4)
    p.add_argument("--max-iter", type=int, default=500)
    p.add_argument("--plain-sample", type=int, default=64)
    p.add_argument("--cpu-iters", type=int, default=20)
    p.add_argument("--no-cpu", action="store_true")
    p.add_argument("--no-plain", action="store_true")
    p.add_argument("--no-e2e", action="store_true")
    p.add_argument("--no-autotune", action="store_true")
    p.add_argument("--no-extras", action="store_true", help="skip the FP32 / double-float / swarm timings")
    p.add_argument("--tpc", type=int, default=0, help="threads per CTA (with --no-autotune)")
    p.add_argument("--variant", type=int, default=0, help="kernel register variant (with --no-autotune)")
    p.add_argument("--cps", type=int, default=0, help="resident CTAs per SM (with --no-autotune; 0 = as many as fit)")
    return p.parse_args()


# ----------------------------------------------------------------------------- clocks
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.idx = gpu_index
        self.proc = None
        self.lines = []

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.idx), f"--query-gpu={self.FIELDS}",
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
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()

    def summary(self):
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx.append(float(f[2]))
            except ValueError:
                continue
            for n, v in zip(names, f[5:9]):
                if v.lower() == "active":
                    reasons.add(n)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"]}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


# ----------------------------------------------------------------------------- helpers
def source_hash() -> str:
    """Hash of the CUDA sources and the C ABI header (what a kernel profile was taken on)."""
    import hashlib
    h = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_2602_15838_gb300", "csrc")
    for name in sorted(os.listdir(csrc)):
        if name.endswith((".cu", ".cuh", ".h")):
            with open(os.path.join(csrc, name), "rb") as f:
                h.update(name.encode() + b"\0" + f.read())
    with open(os.path.join(ROOT, "include", "tadmm.h"), "rb") as f:
        h.update(f.read())
    return h.hexdigest()[:16]


def profile_counters(tpc: int, variant: int):
    """Figures of the committed ncu summary of k_batched (key = value lines) for
    this launch shape, or (None, reason) when the kernel sources or the launch
    shape differ from the profiled ones."""
    try:
        with open(COUNTERS_FILE) as f:
            kv = dict(ln.split("=", 1) for ln in f if "=" in ln and not ln.lstrip().startswith("#"))
    except OSError:
        return None, "no profile summary"
    kv = {k.strip(): v.strip() for k, v in kv.items()}
    if kv.get("source_hash") != source_hash():
        return None, "kernel sources changed since the profile (hash %s, now %s)" % (kv.get("source_hash"),
                                                                                    source_hash())
    variants = [int(v) for v in kv.get("variants", "").split(",") if v.strip()]
    if int(kv.get("threads_per_cta", -1)) != tpc or variant not in variants:
        return None, "launch shape differs from the profiled ones"
    kv["dram_bytes_per_launch"] = kv["variant%d.dram_bytes_per_launch" % variant]
    for key in ("executed_per_algorithmic_flop", "small_case", "executed_per_required_flop", "required_case"):
        kv[key] = kv.get("variant%d.%s" % (variant, key), kv.get(key))
    if kv.get("executed_per_algorithmic_flop") is None:
        return None, "no executed-instruction counts for this variant"
    return kv, None


def measure_fma_peaks(tg, torch, target_ms=40.0):
    """FP64 and FP32 FMA throughput of this GPU (TFLOP/s) from the library's
    probe kernel, timed with CUDA events; best of 3 after a calibration run."""
    import ctypes as C
    L = tg.lib()
    L.tadmm_fma_probe.argtypes = [C.c_int32, C.c_int32, C.c_int32, C.POINTER(C.c_double), C.c_void_p]
    stream = torch.cuda.current_stream()
    sp = C.c_void_p(stream.cuda_stream)
    out = {}
    for prec in (64, 32):
        fl = C.c_double(0.0)

        def timed(iters):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            tg._check(L.tadmm_fma_probe(prec, int(iters), 8, C.byref(fl), sp), "tadmm_fma_probe")
            e1.record(stream)
            torch.cuda.synchronize()
            return e0.elapsed_time(e1), fl.value
        iters = 2000 if prec == 64 else 50000
        ms, _ = timed(iters)
        iters = max(1, int(iters * target_ms / max(ms, 1e-3)))
        best = min(timed(iters)[0] for _ in range(3))
        out[prec] = fl.value / (best / 1e3) / 1e12
    return out


def workload_batch(n_scen: int, rank: int):
    """Rank r's shard of the weak-scaling job: scenario ids r*n_scen .. (r+1)*n_scen-1."""
    from instances import make_workload
    return make_workload("mixed", n_scen=n_scen, first=rank * n_scen)


def aggregate(t_local: float, solves_local: float, dist, device):
    """Whole-job figures over ranks: max of the timed seconds, sum of the solves
    (host-side bookkeeping only; no collective touches the solver's data)."""
    import torch
    if dist is None:
        return t_local, float(solves_local)
    t = torch.tensor([t_local], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    s_ = torch.tensor([float(solves_local)], dtype=torch.float64, device=device)
    dist.all_reduce(s_)
    return float(t.item()), float(s_.item())


def required_flops(batch, cnt, sol, projected=0.0):
    """FP64 flops that one step cannot do without, from the kernel's counters (per-unit
    figures above) and the share of its pair-steps that are projected."""
    fp, fe, ff = FLOPS_2D if batch.nx == 4 else FLOPS_3D
    T = batch.T.astype(np.float64)
    lqr = np.where(sol["iters"] > 0, batch.N, 0) * T   # warm-start LQR solve of the first iteration
    eqp_stages = float((cnt["eqp"] * T).sum() + lqr.sum())
    fact_stages = float(cnt["fact"].sum())
    pairsteps = float(cnt["pairsteps"].sum())
    flops = fp * projected * pairsteps + fe * eqp_stages + ff * fact_stages
    return flops, dict(pairsteps=pairsteps, eqp_stages=eqp_stages, fact_stages=fact_stages)


def cpu_baseline(batch, args, gpu_solves_per_scen_iter):
    """Oracle on a bounded seeded sample; scaled to solves/s."""
    import oracle
    cores = os.cpu_count() or 1
    rng = np.random.default_rng(1234)
    nsamp = min(batch.n_scen, cores)
    idx = sorted(rng.choice(batch.n_scen, nsamp, replace=False).tolist())
    t0 = time.perf_counter()
    res, used = oracle.admm_batch(batch, idx, start_mode=oracle.START_TURBO, tol=0.0, max_iter=args.cpu_iters,
                                  nthreads=cores)
    dt = time.perf_counter() - t0
    scen_iter_per_s = sum(r["iters"] for r in res) / dt
    return dict(value=scen_iter_per_s * gpu_solves_per_scen_iter, unit=UNIT, cores=int(used), kind="oracle",
                sample=f"{nsamp} seeded scenarios of the batch x {args.cpu_iters} ADMM iterations each "
                       f"({dt:.1f} s, {scen_iter_per_s:.2f} scenario-iterations/s), scaled by the GPU run's "
                       f"solves per scenario-iteration")


# ----------------------------------------------------------------------------- reference arm
def run_reference(args, rank, world):
    if rank != 0:
        return
    import oracle
    batch = workload_batch(args.n_scen, 0)
    cores = os.cpu_count() or 1
    nsamp = min(batch.n_scen, cores)
    rng = np.random.default_rng(1234)
    times, iters_done, used = [], 0, 1
    for step in range(args.warmup + args.steps):
        idx = sorted(rng.choice(batch.n_scen, nsamp, replace=False).tolist())
        t0 = time.perf_counter()
        res, used = oracle.admm_batch(batch, idx, start_mode=oracle.START_TURBO, tol=0.0,
                                      max_iter=args.cpu_iters, nthreads=cores)
        dt = time.perf_counter() - t0
        if step >= args.warmup:
            times.append(dt)
            iters_done += sum(r["iters"] for r in res)
    total = sum(times)
    scen_iter_per_s = iters_done / total if total > 0 else 0.0
    value = scen_iter_per_s * WORKLOAD_SOLVES_PER_SCEN_ITER
    sample = (f"per step {nsamp} seeded scenarios of the batch x {args.cpu_iters} ADMM iterations "
              f"({scen_iter_per_s:.2f} scenario-iterations/s), scaled to solves/s by the workload's "
              f"{WORKLOAD_SOLVES_PER_SCEN_ITER:.4e} solves per scenario-iteration")
    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": 1e3 * total / max(1, len(times)), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic", "impl": "reference",
            "config": {"workload": f"mixed batch: {args.n_scen} scenarios, N~U{{2..32}}, T~U{{20..40}}, 2D "
                                   f"double integrator, d_min 0.4, rho 1, |u|<=1; tol {args.tol}, "
                                   f"max_iter {args.max_iter}", "n_scen": args.n_scen},
            "cpu_baseline": {"value": value, "unit": UNIT, "kind": "oracle", "cores": int(used), "sample": sample},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


# ----------------------------------------------------------------------------- our arm
def run_ours(args, rank, world):
    import torch
    import paper_2602_15838_gb300 as tg
    from paper_2602_15838_gb300 import build as tb
    tb.build()

    dev = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(dev)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", dev))

    def barrier():
        if dist is not None:
            dist.barrier()

    batch = workload_batch(args.n_scen, rank)
    solver = tg.Solver(batch, precision=args.precision, start="turbo", mode="batched",
                       threads_per_cta=args.tpc, ctas_per_sm=args.cps, kernel_variant=args.variant)
    tpc, cps, var = (args.tpc, args.cps, args.variant) if args.no_autotune else solver.autotune(probe_iter=100)
    stream = torch.cuda.current_stream()
    peak_clocks = ClockSampler(dev)
    with peak_clocks:
        peaks = measure_fma_peaks(tg, torch)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device="cuda")

    for _ in range(args.warmup):
        solver.solve(args.tol, args.max_iter)
    torch.cuda.synchronize()

    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    clocks = ClockSampler(dev)
    barrier()
    torch.cuda.synchronize()
    with clocks:
        for k in range(args.steps):
            flush.zero_()                       # evict L2 between steps (outside the events)
            ev[k][0].record(stream)
            solver.solve(args.tol, args.max_iter)
            ev[k][1].record(stream)
        torch.cuda.synchronize()
    barrier()
    step_ms = [a.elapsed_time(b) for a, b in ev]
    t_local = sum(step_ms) / 1e3
    sol = solver.solution()
    cnt = solver.counters()
    solves_local = int((sol["status"] == tg.CONVERGED).sum())
    scen_iters = int(sol["iters"].sum())
    t_max, solves_all = aggregate(t_local, solves_local, dist, "cuda")
    value = solves_all * args.steps / t_max if t_max > 0 else 0.0
    ms_step = 1e3 * t_max / args.steps
    headline = (args.n_scen, args.max_iter, args.precision, args.tol) == (4096, 500, 64, 1e-4)
    flops, units = required_flops(batch, cnt, sol, WORKLOAD_PROJECTED_SHARE if headline else 0.0)
    achieved = flops / (t_local / args.steps) / 1e12

    # end to end through the C ABI from pinned host buffers: two handles on two
    # streams, double-buffered, so that step k + 1's upload and solve are enqueued
    # before step k's results are read back (every step still copies all of its
    # inputs in and its results out inside the timed region)
    # the same steps pipelined over two handles on two streams (device-timed, data
    # resident): step k + 1's launch is enqueued behind step k on the other stream,
    # so the tail of one batch, when few scenario groups are left, overlaps the start
    # of the next; reported beside `value`, which times every step in isolation
    second = tg.Solver(batch, precision=args.precision, start="turbo", mode="batched",
                       threads_per_cta=tpc, ctas_per_sm=cps, kernel_variant=var)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    handles = [solver, second]
    for k in range(2):
        with torch.cuda.stream(streams[k]):
            handles[k].solve(args.tol, args.max_iter, stream=streams[k])
    torch.cuda.synchronize()
    p0, p1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    p0.record(streams[0])
    streams[1].wait_event(p0)
    for k in range(args.steps):
        handles[k % 2].solve(args.tol, args.max_iter, stream=streams[k % 2])
    last = torch.cuda.Event()
    last.record(streams[1])
    streams[0].wait_event(last)
    p1.record(streams[0])
    torch.cuda.synchronize()
    pipe_ms = p0.elapsed_time(p1) / args.steps
    pipe_solves = sum(int((h.solution()["status"] == tg.CONVERGED).sum()) for h in handles) / 2.0
    pipelined = {"value": pipe_solves / (pipe_ms / 1e3), "unit": UNIT, "ms_per_step": pipe_ms,
                 "fp64_tflops": flops / (pipe_ms / 1e3) / 1e12, "frac_of_measured_fp64": None,
                 "note": ("device-timed like value, two handles on two streams taking alternate steps (inputs "
                          "resident, each handle's state > L2, no flush): one batch's tail overlaps the next "
                          "batch's start")}

    if peaks.get(64):
        pipelined["frac_of_measured_fp64"] = pipelined["fp64_tflops"] / peaks[64]

    e2e = None
    if not args.no_e2e:
        import ctypes as C
        L = tg.lib()
        hb = tg._HostBatch(batch, pinned=True)
        sps = [C.c_void_p(x.cuda_stream) for x in streams]
        outs = []
        for _ in range(2):
            outs.append(dict(X=torch.empty(solver.sizes["X"], dtype=torch.float64).pin_memory(),
                             U=torch.empty(solver.sizes["U"], dtype=torch.float64).pin_memory(),
                             TH=torch.empty(max(1, solver.sizes["theta"]), dtype=torch.float64).pin_memory(),
                             W=torch.empty(solver.sizes["U"], dtype=torch.int8).pin_memory(),
                             st=torch.empty(batch.n_scen, dtype=torch.int32).pin_memory(),
                             it=torch.empty(batch.n_scen, dtype=torch.int32).pin_memory(),
                             rs=torch.empty(2 * batch.n_scen, dtype=torch.float64).pin_memory()))

        def enqueue(k):
            h, sp = handles[k % 2].h, sps[k % 2]
            tg._check(L.tadmm_update(h, C.byref(hb.s), sp), "tadmm_update")
            tg._check(L.tadmm_solve(h, args.tol, args.max_iter, sp), "tadmm_solve")

        def collect(k):
            o = outs[k % 2]
            tg._check(L.tadmm_get_solution(handles[k % 2].h, *[C.c_void_p(o[n].data_ptr()) for n in
                                                                ("X", "U", "TH", "W", "st", "it", "rs")],
                                           sps[k % 2]), "tadmm_get_solution")
            return int((o["st"].numpy() == 0).sum())

        for k in range(2):            # warm-up: each handle's graph is captured on its first solve
            enqueue(k)
            collect(k)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        enqueue(0)
        e2e_solves = 0
        for k in range(args.steps):
            if k + 1 < args.steps:
                enqueue(k + 1)
            e2e_solves += collect(k)
        e2e_s = time.perf_counter() - t0
        o = outs[0]
        h2d = sum(v.nbytes for v in hb.keep.values()) + hb.N.nbytes + hb.T.nbytes
        d2h = (o["X"].numel() * 8 + o["U"].numel() * 8 + o["TH"].numel() * 8 + o["W"].numel()
               + 4 * 2 * batch.n_scen + 16 * batch.n_scen)
        e2e = {"value": e2e_solves / e2e_s, "unit": UNIT, "h2d_bytes_per_step": int(h2d),
               "d2h_bytes_per_step": int(d2h), "ms_per_step": 1e3 * e2e_s / args.steps,
               "pipeline": "two handles on two streams: step k+1 uploaded and solved while step k is read back"}

    second.close()

    out = None
    if rank == 0:
        plain = None
        if not args.no_plain:
            rng = np.random.default_rng(99)
            idx = sorted(rng.choice(batch.n_scen, min(args.plain_sample, batch.n_scen), replace=False).tolist())
            sub = batch.subset(idx)
            ps = tg.Solver(sub, precision=args.precision, start="turbo", mode="plain")
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            ps.solve(args.tol, args.max_iter)
            torch.cuda.synchronize()
            pdt = time.perf_counter() - t0
            psol = ps.solution()
            pconv = int((psol["status"] == 0).sum())
            pscen_iters = int(psol["iters"].sum())
            ps.close()
            # batched on the same sample, for the work-matched comparison
            bs = tg.Solver(sub, precision=args.precision, start="turbo", mode="batched")
            bs.solve(args.tol, args.max_iter)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            bs.solve(args.tol, args.max_iter)
            torch.cuda.synchronize()
            bdt = time.perf_counter() - t0
            bs.close()
            scen_iter_rate = scen_iters * args.steps / t_local
            plain = {"value": pconv / pdt, "unit": UNIT, "scenarios": len(idx), "solves": pconv,
                     "seconds": pdt, "scenario_iterations_per_s": pscen_iters / pdt,
                     "speedup_scenario_iterations": scen_iter_rate / (pscen_iters / pdt),
                     "batched_same_sample_seconds": bdt,
                     "speedup_batched_full_vs_plain": (value / (pconv / pdt)) if pconv else None,
                     "speedup_same_sample_wall": pdt / bdt,
                     "note": "work-matched speedup = batched scenario-iterations/s over plain; the solves/s "
                             "ratio also reflects which sampled scenarios converge within the cap"}
        cpu = None
        if not args.no_cpu:
            cpu = cpu_baseline(batch, args, solves_local / max(1, scen_iters))
        ext = None if args.no_extras else extras(tg, torch, batch, args, peaks)
        clk = clocks.summary()
        launches = args.steps * solver_launches(solver)
        prof, prof_why = profile_counters(tpc, var)
        traffic = executed = None
        if prof is not None and headline:
            traffic = float(prof["dram_bytes_per_launch"])
            # executed FP64 thread-flops over the required ones, from a capture of the same
            # iterations on fewer scenarios
            if prof.get("executed_per_required_flop"):
                ratio = float(prof["executed_per_required_flop"])
                ex = achieved * ratio
                executed = {"tflops": ex, "frac": ex / peaks[64], "executed_per_required_flop": ratio,
                            "source": "ncu thread-level DFMA (x2), DADD, DMUL counts of k_batched on "
                                      + prof.get("required_case", "fewer scenarios")}
        out = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms_step, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64" if args.precision == 64 else "f32", "data": "synthetic",
            "config": {"workload": f"mixed batch: {args.n_scen} scenarios per GPU, N~U{{2..32}} agents, "
                                   f"T~U{{20..40}}, 2D double integrator, d_min 0.4, rho 1, |u|<=1; "
                                   f"tol {args.tol}, max_iter {args.max_iter}",
                       "n_scen": args.n_scen, "tol": args.tol, "max_iter": args.max_iter,
                       "precision": args.precision, "parallelism": f"replicas x{world} (scenario shards)",
                       "launch": {"threads_per_cta": tpc, "ctas_per_sm": cps, "kernel_variant": var,
                                  "autotuned": not args.no_autotune},
                       "l2": "256 MB buffer written between steps (outside timing); working set > L2"},
            "solves_per_step": solves_all, "scenarios_per_step": args.n_scen * world,
            "ms_per_solve": (1e3 * t_max / args.steps) / max(1.0, solves_all),
            "scenario_iterations_per_s": scen_iters * args.steps / t_local,
            "clocks": clk,
            "roofline": {"bound": "alu", "kernel": "k_batched (FP64 pipe)", "achieved": achieved,
                         "peak": peaks[64], "unit": "TFLOP/s", "frac": achieved / peaks[64],
                         "traffic": traffic, "traffic_note": prof_why,
                         "peak_source": "measured in this run: FP64 FMA probe kernel (tadmm_fma_probe), 8 CTAs "
                                        "of 256 threads per SM, CUDA events, best of 3",
                         "peak_clocks": peak_clocks.summary(),
                         "peak_fp32_measured": peaks[32],
                         "peak_derived": PEAK_FP64_DERIVED_TFLOPS, "frac_of_derived": achieved / PEAK_FP64_DERIVED_TFLOPS,
                         "peak_derived_source": "152 SMs x 4 FP64 flop/clk x 2.07 GHz",
                         "executed": executed,
                         "algorithmic_units": units, "projected_share": WORKLOAD_PROJECTED_SHARE if headline else 0.0,
                         "required_flops_per_step": flops,
                         "note": "achieved counts the FP64 flops that the step cannot do without; executed counts "
                                 "what the kernel executes"},
            "workload_check": {"solves": solves_local, "scenario_iterations": scen_iters,
                               "matches_reference_arm_constant": (solves_local, scen_iters) ==
                               (WORKLOAD_SOLVES, WORKLOAD_SCEN_ITERS) if args.n_scen == 4096 and rank == 0 and
                               (args.tol, args.max_iter, args.precision) == (1e-4, 500, 64) else None},
            "plain_gpu": plain,
            "cpu_baseline": cpu,
            "extras": ext,
            "e2e": e2e,
            "pipelined": pipelined,
            "gpu_launches": launches,
        }
        print(json.dumps(out), flush=True)
    solver.close()
    if dist is not None:
        dist.destroy_process_group()


def timed_solves(tg, torch, batch, args, reps=2, **kw):
    """Device time and solves of one solve of `batch` (after one untimed solve)."""
    do_tune = kw.pop("autotune", True)
    s = tg.Solver(batch, start="turbo", mode=kw.pop("mode", "batched"), **kw)
    tuned = s.autotune(probe_iter=60) if do_tune else None
    s.solve(args.tol, args.max_iter)
    torch.cuda.synchronize()
    ms = []
    for _ in range(reps):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        s.solve(args.tol, args.max_iter)
        e1.record()
        torch.cuda.synchronize()
        ms.append(e0.elapsed_time(e1))
    sol = s.solution()
    s.close()
    conv = int((sol["status"] == 0).sum())
    m = statistics.median(ms)
    return dict(value=conv / (m / 1e3), unit=UNIT, ms_per_step=m, solves_per_step=conv, launch=tuned)


def _event_ms(torch, fn, reps=5, warm=True):
    """Median device time (CUDA events on the current stream) of fn(), after one
    untimed call unless warm is False."""
    if warm:
        fn()
    torch.cuda.synchronize()
    ms = []
    for _ in range(reps):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        fn()
        e1.record()
        torch.cuda.synchronize()
        ms.append(e0.elapsed_time(e1))
    return statistics.median(ms)


def _loss_grad(b, X):
    """Loss sum ||p_it - target_it||^2 (t = 1..T) of the differentiation workload and dl/dX."""
    g = np.zeros_like(X)
    xo = to = 0
    for k in range(b.n_scen):
        N, T = int(b.N[k]), int(b.T[k])
        Xk = X[xo:xo + N * (T + 1) * b.nx].reshape(N, T + 1, b.nx)
        e = Xk[:, 1:, :b.dp] - b.targets[to:to + N * T].reshape(N, T, b.dp)
        gk = np.zeros_like(Xk)
        gk[:, 1:, :b.dp] = 2 * e
        g[xo:xo + gk.size] = gk.ravel()
        xo += gk.size
        to += N * T
    return g


def other_workloads(tg, torch, args, peaks):
    """The remaining synthetic workloads, device-timed with CUDA events."""
    from instances import make_workload
    out = {}
    # 2 agents, T = 20: latency of one solve to tol 1e-4 in each execution mode
    def frac(bb, s, ms):
        fl, _ = required_flops(bb, s.counters(), s.solution())
        return fl / (ms / 1e3) / 1e12 / peaks[64]

    b = make_workload("pair")
    row = {}
    for mode in ("batched", "graph", "plain"):
        s = tg.Solver(b, precision=64, mode=mode)
        row[f"ms_per_solve_{mode}"] = ms = _event_ms(torch, lambda: s.solve(args.tol, args.max_iter), reps=10)
        row[f"frac_of_measured_fp64_{mode}"] = frac(b, s, ms)
        sol = s.split(s.solution())[0]
        s.close()
        row["iterations"], row["status"] = sol["iters"], sol["status"]
    s = tg.Solver(b, precision=32)
    row["ms_per_solve_batched_fp32"] = _event_ms(torch, lambda: s.solve(args.tol, args.max_iter), reps=10)
    s.close()
    row["note"] = ("one scenario: latency-bound; the FP64 fractions (flops of the agents' solves from the run's "
                   "counters over the measured peak) show how little of the GPU a 2-agent problem occupies")
    out["pair_2_agents"] = row
    # 14 agents, T = 20: ms per iteration over 500 iterations; iterations to tol 1e-4 with balancing
    b = make_workload("ring14")
    row = {}
    for mode, prec in (("batched", 64), ("graph", 64), ("plain", 64), ("batched", 32)):
        s = tg.Solver(b, precision=prec, mode=mode)
        ms = _event_ms(torch, lambda: s.solve(0.0, 500), reps=3)
        row[f"ms_per_iteration_{mode}_fp{prec}"] = ms / 500
        if prec == 64:
            row[f"frac_of_measured_fp64_{mode}"] = frac(b, s, ms)
        s.close()
    s = tg.Solver(b, precision=64)
    s.solve(args.tol, args.max_iter)
    sol = s.split(s.solution())[0]
    s.close()
    row["status_at_500"], row["residual_r_at_500"] = sol["status"], sol["r"]
    s = tg.Solver(b, precision=64, adapt=(10, 10.0, 2.0))
    row["ms_to_tol_with_residual_balancing"] = _event_ms(torch, lambda: s.solve(args.tol, 20000), reps=2)
    sol = s.split(s.solution())[0]
    s.close()
    row["iterations_to_tol_with_residual_balancing"], row["status_with_residual_balancing"] = sol["iters"], sol["status"]
    row["note"] = ("rho = 1 as the workload states does not reach 1e-4 within 500 iterations (the oracle agrees); "
                   "residual balancing (every 10 iterations, mu 10, tau 2) is an extension, labelled as such")
    out["ring_14_agents"] = row
    # 512 agents, 3D, T = 40: graph mode, ms per iteration over 100 iterations, FP64 roofline
    b = make_workload("swarm3d")
    row = {}
    s = tg.Solver(b, precision=64, mode="graph")
    ms = _event_ms(torch, lambda: s.solve(0.0, 100), reps=2)
    cnt, sol = s.counters(), s.solution()
    s.close()
    fl, units = required_flops(b, cnt, sol)
    row.update(ms_per_iteration_graph=ms / 100, iterations=100, algorithmic_units_per_100=units,
               tflops=fl / (ms / 1e3) / 1e12, frac_of_measured_fp64=fl / (ms / 1e3) / 1e12 / peaks[64])
    s = tg.Solver(b, precision=64, mode="plain")
    row["ms_per_iteration_plain"] = _event_ms(torch, lambda: s.solve(0.0, 20), reps=2) / 20
    s.close()
    row["note"] = ("one scenario of 130816 pairs x 40 steps; the FP64 fraction counts the agents' solves "
                   "(78 flops per EQP stage, 105 per factorized stage) over the measured FP64 peak")
    out["swarm3d_512_agents"] = row
    # 64 scenarios x 16 agents, T = 30: solve, active-set polish and implicit-KKT backward
    b = make_workload("diff", n_scen=64)
    for prec, tol, iters in ((64, 1e-6, 2000), (32, 1e-5, 5000)):
        row = {}
        s = tg.Solver(b, precision=prec, adapt=(10, 10.0, 2.0))
        row["ms_solve"] = _event_ms(torch, lambda: s.solve(tol, iters), reps=2)
        if prec == 64:
            row["solve_frac_of_measured_fp64"] = frac(b, s, row["ms_solve"])
        t0 = time.perf_counter()
        pol = s.polish(1e-9, 100)
        row["ms_polish"] = 1e3 * (time.perf_counter() - t0)
        row["polish_rounds"], row["polished_to_kkt"] = pol["rounds"], int((pol["status"] == 0).sum())
        gX = _loss_grad(b, s.backward(None)["X_polished"])
        row["ms_backward"] = _event_ms(torch, lambda: s.backward(gX), reps=3)
        s.close()
        row["note"] = (f"ADMM with residual balancing to tol {tol} or {iters} iterations, then active-set "
                       "polishing (host-synchronized rounds, wall time) and the adjoint (host wall time "
                       "includes the copies of the gradients)")
        out[f"differentiation_64x16_fp{prec}"] = row
    return out


def extras(tg, torch, batch, args, peaks):
    out = {}
    out["fp32"] = timed_solves(tg, torch, batch, args, precision=32)
    out["fp32"]["note"] = "float32 arithmetic, same workload; parity 1e-4 against the float64 oracle"
    out["double_float"] = timed_solves(tg, torch, batch, args, precision=64, flags=tg.FLAG_DOUBLE_FLOAT)
    out["double_float"]["note"] = "float64-grade double-float arithmetic on the FP32 pipe (parity 1e-9)"
    out["residual_balancing"] = timed_solves(tg, torch, batch, args, precision=64, adapt=(10, 10.0, 2.0))
    out["residual_balancing"]["note"] = ("rho balanced every 10 iterations (mu 10, tau 2; Boyd et al. 2011, "
                                         "Sec. 3.4.1), an extension beyond the fixed rho = 1 of the workload; "
                                         "parity against the oracle's balancing 1e-9")
    out["balancing_relaxed"] = timed_solves(tg, torch, batch, args, precision=64, adapt=(10, 10.0, 2.0), relax=1.6)
    out["balancing_relaxed"]["note"] = ("residual balancing as above plus over-relaxation alpha = 1.6 (Boyd et al. "
                                        "2011, Sec. 3.4.3), an extension; parity against the oracle 1e-9")
    from instances import heterogeneous_agents, nearest_neighbour_pairs
    out["heterogeneous_agents"] = timed_solves(tg, torch, heterogeneous_agents(batch, seed=7), args, precision=64)
    out["heterogeneous_agents"]["note"] = ("per-agent dynamics (seeded velocity damping and mass per agent, "
                                           "recursions by axis) on the same workload, an extension; parity 1e-9")
    knn = nearest_neighbour_pairs(batch, 4)
    out["knn_coupling"] = timed_solves(tg, torch, knn, args, precision=64)
    out["knn_coupling"]["note"] = ("listed pairs: each agent coupled to its 4 nearest agents at t = 0 (%d of %d "
                                   "pairs), an extension; parity 1e-9" % (int(knn.pair_count.sum()), int(batch.P.sum())))
    # one outer linearize-and-solve step: the device-side re-linearization of every halfspace
    s = tg.Solver(batch, precision=64)
    s.solve(args.tol, 20)
    ms = _event_ms(torch, s.relinearize, reps=3)
    s.close()
    out["relinearize"] = {"ms": ms, "pair_steps": int((batch.P * batch.T).sum()),
                          "note": "normals and guesses re-formed at the last iterate, whole batch, one call"}
    out["sqp_loop"] = sqp_loop(tg, torch, batch, args)
    out.update(other_workloads(tg, torch, args, peaks))
    out["homotopy_hot_start"] = homotopy_vs_primal(tg, torch, batch)
    out["start_mode_ablation"] = start_mode_ablation(tg, torch, args)
    return out


def sqp_loop(tg, torch, batch, args, max_outer=6):
    """The linearize-and-solve loop with the termination rule of Sec. V.A
    (relative objective change <= 1e-4 between outer steps, collision-free up to
    the solve's tolerance) on the whole batch under residual balancing: wall
    time of the loop (it synchronizes after every outer step), outer steps per
    scenario and how many met the rule (only scenarios whose ADMM solve
    converged can)."""
    s = tg.Solver(batch, precision=64, adapt=(10, 10.0, 2.0))
    tuned = s.autotune(probe_iter=60)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    r = s.sqp(tol=args.tol, max_iter=args.max_iter, max_outer=max_outer, obj_rtol=1e-4)
    wall = 1e3 * (time.perf_counter() - t0)
    s.close()
    met = r["status"] == 0
    steps = np.bincount(r["outer"][met], minlength=max_outer + 1)[1:].tolist()
    return {"ms_wall": wall, "launch": tuned, "max_outer": max_outer, "scenarios": int(batch.n_scen), "met_rule": int(met.sum()),
            "outer_steps_of_those": steps,
            "min_dist_over_d_min_of_those": float((r["min_dist"][met] / batch.d_min[met]).min()) if met.any() else None,
            "note": ("every outer step solves the whole batch (scenarios that met the rule keep their data); "
                     "tol %g, %d ADMM iterations per solve, residual balancing (mu 10, tau 2 every 10), "
                     "an extension beyond the single linearized QP" % (args.tol, args.max_iter))}


def start_mode_ablation(tg, torch, args):
    """The paper's ablation (BaseADMM = cold start every iteration, HotstartADMM =
    hot start, TurboADMM = affine-LQR warm start then hot start) over the paper's
    agent counts 2, 4, 6, 10 and 14 (the 2-agent crossing and the ring of N agents
    on a radius-5 circle with antipodal goals): device time, ADMM iterations and
    active-set EQP solves summed over agents and iterations (the paper's table
    counts the per-agent QP iterations the same way).  Two settings: graph mode at
    the workload's fixed rho = 1 to tol 1e-4 or 500 iterations, and the batched
    kernel with residual balancing (an extension) to tol 1e-4 or 5000 iterations,
    where every start converges."""
    from instances import make_workload
    out = {}
    for N in (2, 4, 6, 10, 14):
        b = make_workload("pair") if N == 2 else make_workload("ring14", N_override=N)
        row = {}
        for setting, kw, iters in (("fixed_rho_graph", dict(mode="graph"), args.max_iter),
                                   ("balanced_batched", dict(mode="batched", adapt=(10, 10.0, 2.0)), 5000)):
            cell = {}
            for label, start in (("base_cold", "cold"), ("hotstart", "hot"), ("turbo", "turbo")):
                s = tg.Solver(b, precision=64, start=start, **kw)
                if start == "cold":      # seconds long: one short untimed solve prepares the launch, one timed
                    s.solve(args.tol, 2)
                    ms = _event_ms(torch, lambda: s.solve(args.tol, iters), reps=1, warm=False)
                else:
                    ms = _event_ms(torch, lambda: s.solve(args.tol, iters), reps=3)
                sol = s.split(s.solution())[0]
                cell[label] = {"ms": ms, "iterations": sol["iters"], "status": sol["status"],
                               "eqp_solves": int(s.counters()["eqp"][0])}
                s.close()
            row[setting] = cell
        out["pair" if N == 2 else f"ring_{N}"] = row
    out["note"] = ("same instances and tolerance for every start; the per-agent QP solution is unique, so the "
                   "iterates agree and only the active-set work differs; the GPU's EQP counts equal the "
                   "oracle's (tested)")
    return out


def homotopy_vs_primal(tg, torch, batch, iters=100):
    """The parametric (homotopy) hot start against the primal hot start on the
    same batch, both in graph mode (per-phase kernels; the homotopy runs only
    there), the first `iters` ADMM iterations: device time and EQP solves."""
    row = {}
    for start in ("turbo", "homotopy"):
        s = tg.Solver(batch, precision=64, start=start, mode="graph")
        ms = _event_ms(torch, lambda: s.solve(0.0, iters), reps=2)
        cnt = s.counters()
        s.close()
        row[start] = {"ms": ms, "eqp_solves": int(cnt["eqp"].sum()), "factorized_stages": int(cnt["fact"].sum())}
    row["iterations"] = iters
    row["homotopy_over_primal_time"] = row["homotopy"]["ms"] / row["turbo"]["ms"]
    row["note"] = ("graph mode, float64, tol 0; eqp_solves counts the homotopy's direction solves with the "
                   "confirming passes; same iterates either way (the per-agent QP solution is unique)")
    return row


def solver_launches(solver) -> int:
    return 1   # one persistent kernel per step (the graph also holds one memset node)


def main():
    args = parse()
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    if args.impl == "reference":
        run_reference(args, rank, world)
    else:
        run_ours(args, rank, world)


if __name__ == "__main__":
    main()
