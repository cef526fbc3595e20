#!/usr/bin/env python
"""Replica-exchange LJ MD throughput on GB300: replica·atom-steps/s and exch/s.

Default workload (one GPU): 64 replicas x 864 atoms, reduced density 0.8442,
temperatures geometric 0.7-2.0, exchange stride N_x = 10, Verlet skin 0.3,
rc = 2.5, dt = 0.005, SVR tau 0.5, FCC start; mixed-precision batched path.
One bench step = every replica advances N_x MD steps (one persistent launch)
+ one exchange attempt (one launch).  The plain FP64 one-replica-per-launch
path is timed on the same workload for comparison.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference] [--config c1]

Under torchrun each rank runs its own ensemble (different seed, no data-path
collective): weak scaling.  --impl reference times the FP64 CPU oracle on the
host cores instead (rank 0 only).
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from paper_0812_1633_gb300 import inputs  # noqa: E402

CONFIGS = {
    # name: (description, list of ensembles (N, R, t_min, t_max), nx, skin, budget mode,
    # precision); skin "auto": chosen by measurement (paper_0812_1633_gb300.tune)
    "c0": ("8 replicas x 256 atoms, rho 0.8442, T 0.8-1.6 geometric, N_x 100",
           [(256, 8, 0.8, 1.6)], 100, 0.5, "fixed", "fp64"),
    "c1": ("64 replicas x 864 atoms, rho 0.8442, T 0.7-2.0 geometric, N_x 10, skin 0.3",
           [(864, 64, 0.7, 2.0)], 10, 0.3, "fixed", "mixed"),
    "c2": ("5 ensembles in one launch: 16x256, 32x500, 48x864, 64x2048, 96x4000 atoms, T 0.7-2.5, "
           "budgets uniform 5-50 per replica per attempt",
           [(256, 16, 0.7, 2.5), (500, 32, 0.7, 2.5), (864, 48, 0.7, 2.5), (2048, 64, 0.7, 2.5),
            (4000, 96, 0.7, 2.5)], 0, "auto", "random", "mixed"),
    "c3": ("256 replicas x 4000 atoms, rho 0.8442, T 0.75-1.8 geometric, N_x 10",
           [(4000, 256, 0.75, 1.8)], 10, 0.5, "fixed", "mixed"),
    "c4": ("1024 replicas x 2048 atoms, rho 0.8442, T 0.7-3.0 geometric, N_x 1",
           [(2048, 1024, 0.7, 3.0)], 1, "auto", "fixed", "mixed"),
}
FLOPS_PER_PAIR = 37.0   # unique pair: 34 for the pair itself + 3 for the reaction
FP32_PEAK_TFLOPS = 152 * 128 * 2 * 2.070e9 / 1e12   # SMs x FP32 lanes x FMA x max SM clock
FP64_PEAK_TFLOPS = 1.25   # nominal GB300 FP64 rate (no measured FP64 peak is provided)


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def rank_seed(rank):
    """Each rank runs its own ensemble: a distinct seed per rank (weak scaling)."""
    return 12345 + 1 + 1000 * rank


def aggregate(total_s, work, ws, dist=None):
    """Whole-job throughput: the slowest rank's time (max over ranks) and the
    sum of the ranks' work (every rank runs the same workload)."""
    if dist is not None and ws > 1:
        import torch
        t = torch.tensor([total_s], dtype=torch.float64)
        w = torch.tensor([work], dtype=torch.float64)
        if dist.get_backend() == "nccl":
            t, w = t.cuda(), w.cuda()
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        dist.all_reduce(w, op=dist.ReduceOp.SUM)
        total_s, work = float(t.item()), float(w.item())
    else:
        work = work * ws
    return total_s, work / total_s


def oracle_skin(cfg):
    """The oracle's skin for a workload: its own, or 0.5 (the paper's list
    radius 3.0) where the GPU path chooses it by measurement."""
    return 0.5 if cfg[3] == "auto" else cfg[3]


def make_budgets(cfg, R, cycles, seed):
    _, ens, nx, _, mode, _ = cfg
    if mode == "random":
        return inputs.random_budgets(R, cycles, 5, 50, seed)
    return np.full((cycles, R), nx, dtype=np.int32)


def atoms_per_cycle(cfg, budgets_row):
    Ns = np.concatenate([[N] * R for (N, R, _, _) in cfg[1]])
    return float((Ns * budgets_row).sum())


# ------------------------------------------------------------------ oracle legs
def oracle_rate(cfg, seed, wall_target=10.0, max_steps=2000):
    """Replica·atom-steps/s of the FP64 CPU oracle on this host's cores."""
    import oracle as O
    nthreads = os.cpu_count() or 1
    ens_list = []
    for i, (N, R, t0, t1) in enumerate(cfg[1]):
        L = inputs.box_length(N)
        ens_list.append(O.Ensemble(N, L, inputs.geometric_ladder(t0, t1, R), seed + i, skin=oracle_skin(cfg)))
    steps = 2
    done_atoms, spent = 0.0, 0.0
    while True:
        t0 = time.perf_counter()
        for e in ens_list:
            e.advance([steps] * e.R, nthreads=nthreads)
        dt = time.perf_counter() - t0
        done_atoms += steps * sum(e.R * e.reps[0].N for e in ens_list)
        spent += dt
        if spent >= wall_target or steps >= max_steps:
            break
        steps = int(min(max_steps, max(steps * 2, steps * wall_target / max(dt, 1e-3) * 0.5)))
    sample = (f"{'+'.join(f'{e.R}x{e.reps[0].N}' for e in ens_list)} replicas x atoms, "
              f"{int(done_atoms / sum(e.R * e.reps[0].N for e in ens_list))} MD steps each from the "
              f"FCC start, {spent:.1f} s wall")
    return done_atoms / spent, nthreads, sample


def run_reference(args, cfg):
    ws, rank, _ = dist_env()
    if rank != 0:
        return
    import oracle as O
    nthreads = os.cpu_count() or 1
    seed = 12345 + 1
    ens_list = []
    for i, (N, R, t0, t1) in enumerate(cfg[1]):
        L = inputs.box_length(N)
        ens_list.append(O.Ensemble(N, L, inputs.geometric_ladder(t0, t1, R), seed + i, skin=oracle_skin(cfg)))
    Rtot = sum(e.R for e in ens_list)
    # each reference step: the whole workload's cycle for small configs; a
    # bounded sample of replicas for large ones (size-normalised metric)
    cap_atoms = 600_000
    sub = []
    for e in ens_list:
        k = max(1, min(e.R, cap_atoms // max(1, e.reps[0].N * len(ens_list))))
        sub.append(k)
    budgets = make_budgets(cfg, Rtot, args.warmup + args.steps, 7)
    times, work = [], 0.0
    for c in range(args.warmup + args.steps):
        off = 0
        t0 = time.perf_counter()
        w = 0.0
        for e, k in zip(ens_list, sub):
            b = budgets[c][off:off + e.R].copy()
            b[k:] = 0
            e.advance(b, nthreads=nthreads)
            e.exchange()
            w += float(b.sum()) * e.reps[0].N
            off += e.R
        dt = time.perf_counter() - t0
        if c >= args.warmup:
            times.append(dt)
            work += w
    total = sum(times)
    value = work / total
    line = {
        "impl": "reference", "metric": "replica·atom-steps/s", "value": value,
        "unit": "replica·atom-steps/s", "n_gpus": ws, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": 1e3 * total / len(times), "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic (FCC start, seeded Philox velocities)",
        "config": {"workload": cfg[0], "replicas_timed": sub},
        "cpu_baseline": {"value": value, "unit": "replica·atom-steps/s", "cores": nthreads,
                         "kind": "oracle",
                         "sample": f"per step: {'+'.join(str(k) for k in sub)} replicas of the workload "
                                   f"advance their stride and attempt one exchange"},
        "e2e": {"value": value, "unit": "replica·atom-steps/s", "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


# ------------------------------------------------------------------ clocks
class Clocks:
    """SM clock and throttle reasons sampled every ~1 ms during the timed region
    through NVML (read-only queries via ctypes); nvidia-smi polling as fallback."""
    REASONS = {0x4: "sw_power_cap", 0x8: "hw_slowdown", 0x20: "sw_thermal_slowdown",
               0x40: "hw_thermal_slowdown", 0x80: "hw_power_brake_slowdown"}

    def __init__(self, cuda_index):
        import ctypes as C
        import threading
        self.C, self.threading = C, threading
        self.samples, self.reasons, self.max_mhz = [], set(), None
        self.nvml = self.h = None
        try:
            import torch
            bus = torch.cuda.get_device_properties(cuda_index).pci_bus_id
        except Exception:
            bus = None
        try:
            nv = C.CDLL("libnvidia-ml.so.1")
            if nv.nvmlInit_v2() == 0:
                h = C.c_void_p()
                ok = -1
                if bus:
                    ok = nv.nvmlDeviceGetHandleByPciBusId_v2(bus.encode(), C.byref(h))
                if ok != 0:
                    ok = nv.nvmlDeviceGetHandleByIndex_v2(C.c_uint(cuda_index), C.byref(h))
                if ok == 0:
                    self.nvml, self.h = nv, h
                    m = C.c_uint()
                    if nv.nvmlDeviceGetMaxClockInfo(h, 1, C.byref(m)) == 0:
                        self.max_mhz = float(m.value)
        except OSError:
            pass

    def _poll(self):
        C = self.C
        mhz, rs = C.c_uint(), C.c_ulonglong()
        get_r = getattr(self.nvml, "nvmlDeviceGetCurrentClocksEventReasons", None) or \
            self.nvml.nvmlDeviceGetCurrentClocksThrottleReasons
        while not self.stop.is_set():
            if self.nvml.nvmlDeviceGetClockInfo(self.h, 1, C.byref(mhz)) == 0:
                self.samples.append(float(mhz.value))
            if get_r(self.h, C.byref(rs)) == 0:
                for bit, name in self.REASONS.items():
                    if rs.value & bit:
                        self.reasons.add(name)
            time.sleep(0.001)

    def __enter__(self):
        if self.nvml is not None:
            self.stop = self.threading.Event()
            self.t = self.threading.Thread(target=self._poll, daemon=True)
            self.t.start()
        return self

    def __exit__(self, *a):
        if self.nvml is not None:
            self.stop.set()
            self.t.join()

    def summary(self):
        if self.nvml is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["NVML unavailable"]}
        if not self.samples:
            return {"sm_mhz": None, "sm_max_mhz": self.max_mhz, "reasons": ["no samples"]}
        return {"sm_mhz": statistics.median(self.samples), "sm_max_mhz": self.max_mhz,
                "reasons": sorted(self.reasons), "samples": len(self.samples),
                "source": "NVML, 1 ms period, during the timed steps"}


# ------------------------------------------------------------------ GPU arm
def in_cutoff_pairs_per_atom(x, cfg, n_sample=8, rc=2.5):
    """Mean unique in-cutoff pairs per atom over a sample of replicas (from a state)."""
    tot_pairs = tot_atoms = 0
    off = 0
    for (N, R, _, _) in cfg[1]:
        L = inputs.box_length(N)
        for r in range(min(R, n_sample)):
            p = x[off + r * N: off + (r + 1) * N]
            cnt = 0
            for i0 in range(0, N, 512):
                d = p[None, :, :] - p[i0:i0 + 512, None, :]
                d -= L * np.rint(d / L)
                r2 = (d * d).sum(-1)
                cnt += int((r2 < rc * rc).sum()) - min(512, N - i0)
            tot_pairs += cnt / 2
            tot_atoms += N
        off += N * R
    return tot_pairs / tot_atoms


def equilibrate(ctx, steps, chunk=100):
    """Untimed MD from the FCC start, no exchanges: the timed cycles then see
    the liquid's list-rebuild rate rather than that of the lattice's first
    steps (at N_x = 1 on the 1024 x 2048 workload the first hundred steps run
    about 15 % faster than the liquid)."""
    done = 0
    while done < steps:
        n = min(chunk, steps - done)
        ctx.advance(n)
        done += n


def run_gpu(args, cfg):
    import torch
    import paper_0812_1633_gb300 as re
    from paper_0812_1633_gb300 import build
    ws, rank, local = dist_env()
    torch.cuda.set_device(local)
    dist = None
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    # one rank per node compiles (when the library is out of date); the others
    # wait, so that no two processes write the same object files
    if local == 0:
        build.build()
    if dist is not None:
        dist.barrier()
    re.lib()
    desc, ens_spec, nx, skin, mode, prec = cfg
    seed = rank_seed(rank)
    stream = torch.cuda.current_stream()

    def make(skin_, **kw):
        members = []
        for i, (N, R, t0, t1) in enumerate(ens_spec):
            L = inputs.box_length(N)
            members.append(re.Context(N, L, 2.5, inputs.geometric_ladder(t0, t1, R), seed + i,
                                      skin=skin_, precision=prec, nx=max(nx, 1), **kw))
        c = members[0] if len(members) == 1 else re.Context.group(members)
        if len(members) > 1:
            for m in members:
                m.close()
        c.set_stream(stream)
        equilibrate(c, args.equil_steps)
        return c

    skin_trials = None
    if skin == "auto" and not args.launch:
        from paper_0812_1633_gb300 import tune
        Rtot0 = sum(R for (_, R, _, _) in ens_spec)
        # the same budgets on every rank, and each candidate's time agreed as the
        # slowest rank's: every rank keeps the same skin (one workload)
        tb = make_budgets(cfg, Rtot0, 20, 99) if mode == "random" else None
        agree = None
        if dist is not None:
            def agree(ms):
                t = torch.tensor([ms], dtype=torch.float64, device="cuda")
                dist.all_reduce(t, op=dist.ReduceOp.MAX)
                return float(t.item())
        skin, ctx, skin_trials = tune.choose_skin(make, cycles=20, budgets=tb, agree=agree)
        tuned = ctx.config()
    elif args.launch:
        skin = 0.5 if skin == "auto" else skin
        cl, at, cd = (int(v) for v in args.launch.split(","))
        ctx = make(skin, cluster=cl, atom_threads=at, cell_div=cd, wide_launch=args.wide)
        tuned = ctx.config()
    else:
        ctx = make(skin)
        tuned = ctx.autotune(steps=nx if nx > 0 else 40)  # as the cycles run it
    Rtot = ctx.n_rep
    W, K = args.warmup, args.steps
    budgets = make_budgets(cfg, Rtot, W + K, 7 + rank)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device="cuda")

    def cycle(c):
        ctx.advance(budgets[c])
        ctx.exchange()

    for c in range(W):
        cycle(c)
    torch.cuda.synchronize()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True),
           torch.cuda.Event(enable_timing=True)) for _ in range(K)]
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    with Clocks(local) as clk:
        for k in range(K):
            flush.zero_()   # L2 flush between timed steps (outside the timed events)
            e0, e1, e2 = ev[k]
            e0.record(stream)
            ctx.advance(budgets[W + k])
            e1.record(stream)
            ctx.exchange()
            e2.record(stream)
        torch.cuda.synchronize()
    if dist:
        dist.barrier()
    step_ms = [a.elapsed_time(c) for a, b, c in ev]
    adv_ms = [a.elapsed_time(b) for a, b, c in ev]
    exch_ms = [b.elapsed_time(c) for a, b, c in ev]
    total_s = sum(step_ms) / 1e3
    work = sum(atoms_per_cycle(cfg, budgets[W + k]) for k in range(K))
    total_s, value = aggregate(total_s, work, ws, dist)
    n_ens = len(ens_spec)
    exch_per_s = ws * n_ens * K / total_s
    # pairs per attempt: (R - p) // 2 for first-pair offset p, alternating 0, 1
    pairs_per_attempt = sum((R - p) // 2 for (N, R, _, _) in ens_spec for p in range(2)) / 2

    # ---- roofline of the dominant kernel (the batched MD launch)
    x, _ = ctx.get_state()
    pairs = in_cutoff_pairs_per_atom(x, cfg)
    adv_mean_s = statistics.mean(adv_ms) / 1e3
    flops_per_launch = FLOPS_PER_PAIR * pairs * work / K
    achieved = flops_per_launch / adv_mean_s / 1e12
    peak = FP64_PEAK_TFLOPS if prec == "fp64" else FP32_PEAK_TFLOPS

    # ---- e2e: the public API with host buffers every cycle.  re_run_record
    # copies each cycle's budgets host -> device (pinned) and each cycle's
    # record (partners, accepted flags, T, U, K, econs) device -> host on copy
    # streams beside the compute stream, all of it as one CUDA graph; the call
    # returns once the last record is on the host.  One untimed call first
    # sizes its buffers and captures the graph, which the timed call replays.
    nE = max(3, min(K, 100))
    bE = np.stack([budgets[W + (k % K)] for k in range(nE)])
    ctx.run_record(nE, bE, graph=True)
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    t_e2e0 = time.perf_counter()
    ctx.run_record(nE, bE, graph=True)
    t_e2e = time.perf_counter() - t_e2e0
    e2e_work = sum(atoms_per_cycle(cfg, bE[k]) for k in range(nE))
    _, e2e_value = aggregate(t_e2e, e2e_work, ws, dist)  # slowest rank's time, all ranks' work
    h2d = 4 * Rtot
    d2h = (37 * Rtot + 7) // 8 * 8   # one record row: 4 doubles, an int32 and a byte per replica

    # ---- the same cycles replayed as one captured CUDA graph (re_run with a
    # graph): the host enqueues one graph instead of two launches per cycle
    graph = None
    if mode == "fixed" and args.graph_cycles > 0:
        nG = args.graph_cycles
        ctx.run(nG, graph=True)          # capture and a first, untimed replay
        torch.cuda.synchronize()
        ge0, ge1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        ge0.record(stream)
        ctx.run(nG, graph=True)
        ge1.record(stream)
        torch.cuda.synchronize()
        g_s = ge0.elapsed_time(ge1) / 1e3
        g_work = nG * atoms_per_cycle(cfg, np.full(Rtot, max(nx, 1)))
        g_s, g_value = aggregate(g_s, g_work, ws, dist)
        graph = {"value": g_value, "unit": "replica·atom-steps/s", "cycles": nG,
                 "ms_per_step": 1e3 * g_s / nG, "eager_ms_per_step": 1e3 * total_s / K,
                 "saved_ms_per_step": 1e3 * (total_s / K - g_s / nG),
                 "l2": "not flushed inside the graph (the eager steps flush it)"}

    # ---- the asynchronous scheme (Implementation section) on the same workload:
    # one free-running launch, exchanges decided inside it by the rotating
    # master after N_x of its own steps; no replica waits for the slowest
    free = None
    if args.free_attempts > 0:
        nxf = max(nx, 1)
        ft_local = fwork_local = dsum = 0.0
        why = None
        try:
            ctx.run_free(2, nxf)
            torch.cuda.synchronize()
            s0 = ctx.counters()[0].astype(np.float64)
            fe0, fe1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            fe0.record(stream)
            ctx.run_free(args.free_attempts, nxf)
            fe1.record(stream)
            torch.cuda.synchronize()
            dsteps = ctx.counters()[0].astype(np.float64) - s0
            Ns = np.concatenate([[N] * R for (N, R, _, _) in ens_spec])
            ft_local, fwork_local = fe0.elapsed_time(fe1) / 1e3, float((Ns * dsteps).sum())
            dsum = float(dsteps.sum())
        except re.REError as e:
            why = str(e)
        # every rank reaches this collective: all of them go on, or none
        failed = why is not None
        if dist is not None and ws > 1:
            flag = torch.tensor([1.0 if failed else 0.0], dtype=torch.float64)
            if dist.get_backend() == "nccl":
                flag = flag.cuda()
            dist.all_reduce(flag, op=dist.ReduceOp.MAX)
            failed = flag.item() > 0
        if failed:
            free = {"unavailable": why or "free-running launch refused on another rank"}
        else:
            ft, fval = aggregate(ft_local, fwork_local, ws, dist)
            free = {"value": fval, "unit": "replica·atom-steps/s",
                    "mode": "free-running: one launch, in-launch exchanges (rotating master)",
                    "attempts": args.free_attempts, "nx": nxf,
                    "exch_per_s": ws * len(ens_spec) * args.free_attempts / ft,
                    "mean_steps_per_attempt": dsum / (Rtot * args.free_attempts)}

    # ---- plain FP64 one-replica-per-launch path on the same workload (bounded)
    plain = None
    if len(ens_spec) == 1 and rank == 0 and not args.no_plain:
        N, R, t0, t1 = ens_spec[0]
        L = inputs.box_length(N)
        p = re.Context(N, L, 2.5, inputs.geometric_ladder(t0, t1, R), seed, skin=skin,
                       path="plain", nx=max(nx, 1))
        p.set_stream(stream)
        p.advance(budgets[0])
        p.exchange()
        torch.cuda.synchronize()
        pe0, pe1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        nP = 20  # cycles (about 1.6 s on the 64 x 864 workload)
        pe0.record(stream)
        for k in range(nP):
            p.advance(budgets[W + (k % K)])
            p.exchange()
        pe1.record(stream)
        torch.cuda.synchronize()
        pt = pe0.elapsed_time(pe1) / 1e3
        pw = sum(atoms_per_cycle(cfg, budgets[W + (k % K)]) for k in range(nP))
        plain = {"value": pw / pt, "unit": "replica·atom-steps/s", "steps": nP,
                 "speedup_of_batched_mixed": value / ws / (pw / pt)}
        p.close()

    cpu = None
    if rank == 0 and ws == 1 and not args.no_cpu_baseline:
        rate, cores, sample = oracle_rate(cfg, seed, wall_target=args.cpu_seconds)
        cpu = {"value": rate, "unit": "replica·atom-steps/s", "cores": cores, "kind": "oracle",
               "sample": sample}

    if rank == 0:
        clocks = clk.summary()
        line = {
            "metric": "replica·atom-steps/s", "value": value, "unit": "replica·atom-steps/s",
            "n_gpus": ws, "steps": K, "warmup": W, "ms_per_step": 1e3 * total_s / K,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64" if prec == "fp64" else "f32+f64",
            "data": "synthetic (FCC start at rho 0.8442, seeded Philox velocities and budgets)",
            "config": {"workload": desc, "path": f"{prec} batched (one persistent launch per cycle)",
                       "l2": "flushed between timed steps (256 MB write)",
                       "equilibration": f"{args.equil_steps} untimed MD steps from the FCC start "
                                        f"before tuning and timing",
                       "launch": tuned, "parallelism": f"replicas, {ws} independent ensemble(s)",
                       "skin": skin, "skin_trials_ms_per_cycle": skin_trials},
            "exch_per_s": exch_per_s,
            "pair_attempts_per_s": exch_per_s * pairs_per_attempt / max(n_ens, 1),
            "advance_ms": statistics.mean(adv_ms), "exchange_ms": statistics.mean(exch_ms),
            "roofline": {"bound": "alu", "achieved": achieved, "peak": peak,
                         "unit": "TFLOP/s", "frac": achieved / peak,
                         "traffic": profiled_traffic(args.config, tuned, prec),
                         "ncu_pipes": (profiled_record(args.config, tuned, prec) or {}).get("pipes"),
                         "kernel": f"md_batched_kernel<{prec}>",
                         "peak_source": "FP64 nominal 1.25 TFLOP/s" if prec == "fp64" else
                                        "152 SMs x 128 FP32 lanes x 2 x 2.07 GHz",
                         "algorithmic": f"{FLOPS_PER_PAIR:.0f} flop x {pairs:.2f} unique in-cutoff "
                                        f"pairs per atom-step"},
            "plain_fp64": plain,
            "cpu_baseline": cpu,
            "e2e": {"value": e2e_value, "unit": "replica·atom-steps/s",
                    "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h, "cycles": nE,
                    "call": "re_run_record (budgets in, per-cycle record out; one CUDA graph, "
                            "captured in an untimed call)"},
            "async": free,
            "graph": graph,
            # per step: the advance (one launch, or the ranking kernel and the
            # two classes of a split launch) and the exchange
            "gpu_launches": (4 if tuned.get("wide_n") else 2) * K,
            "clocks": clocks,
        }
        print(json.dumps(line), flush=True)
    ctx.close()
    if dist:
        dist.barrier()
        dist.destroy_process_group()


# ------------------------------------------------------------------ drift study
def drift_slopes(times, H, N):
    """Least-squares slope of H~/N against time (tau) for every replica."""
    t = np.asarray(times)
    Hn = np.asarray(H) / N
    tc = t - t.mean()
    return (tc[:, None] * (Hn - Hn.mean(0))).sum(0) / (tc * tc).sum()


def run_drift(args):
    """Energy drift of H~ = U + K + econs (per atom per tau) for the mixed and
    FP64 batched paths and the plain FP64 path on the same seeded systems
    (the 256-replica precision workload reduced to R replicas); the oracle's
    drift on the same systems comes from tests/parity_report.py."""
    import torch
    import paper_0812_1633_gb300 as re
    from paper_0812_1633_gb300 import build
    build.build()
    N, R = args.drift_n, args.drift_r
    L = inputs.box_length(N)
    temps = inputs.geometric_ladder(0.75, 1.8, R)
    dt, chunk = 0.005, 100
    out = {"study": "energy drift of H~ per atom per tau (least-squares slope)",
           "workload": f"{R} replicas x {N} atoms, rho 0.8442, T 0.75-1.8, dt 0.005, tau_T 0.5, "
                       f"FCC start, seed 12345",
           "steps": args.drift_steps}
    for name, kw in [("mixed_batched", dict(precision="mixed")),
                     ("fp64_batched", dict(precision="fp64")),
                     ("plain_fp64", dict(path="plain"))]:
        steps = args.drift_steps if name != "plain_fp64" else min(args.drift_steps, 4000)
        ctx = re.Context(N, L, 2.5, temps, 12345, **kw)
        t, H = [], []
        t0 = time.perf_counter()
        for c in range(steps // chunk):
            ctx.advance(chunk)
            H.append(ctx.energies()[2])
            t.append((c + 1) * chunk * dt)
        wall = time.perf_counter() - t0
        sl = drift_slopes(t, H, N)
        common = min(len(t), args.drift_window // chunk)
        sc = drift_slopes(t[:common], H[:common], N)
        out[name] = {"mean": float(sl.mean()), "max_abs": float(np.abs(sl).max()),
                     "steps": steps, "replica_atom_steps_per_s": R * N * steps / wall,
                     "common_window": {"steps": common * chunk, "mean": float(sc.mean()),
                                       "max_abs": float(np.abs(sc).max())}}
        ctx.close()
    out["oracle"] = "measured by tests/parity_report.py (the oracle is test infrastructure)"
    print(json.dumps(out), flush=True)


# The precision study of the 256 x 4000 workload (T 0.75-1.8): its 16 coldest
# replicas (consecutive on the 256-replica ladder), N = 4000, FCC start.
PREC_N, PREC_R, PREC_SEED = 4000, 16, 12345


def precision_temps():
    return inputs.geometric_ladder(0.75, 1.8, 256)[:PREC_R]


def drift_run(ctx, steps, chunk, N, dt=0.005, budgets=None):
    """H~/N sampled every `chunk` steps; returns the least-squares slope per
    replica (per atom per tau) and the wall time."""
    t, H = [], []
    t0 = time.perf_counter()
    for c in range(steps // chunk):
        ctx.advance(chunk if budgets is None else budgets * chunk)
        H.append(ctx.energies()[2])
        t.append((c + 1) * chunk * dt)
    return drift_slopes(t, H, N), time.perf_counter() - t0


def exchange_run(ctx, cycles, nx, N, dt=0.005, sample=10):
    """cycles x (advance nx, exchange): acceptance per ladder pair and H~ slope
    (H~ stays continuous across exchanges)."""
    att0, acc0 = ctx.accept_stats()
    t, H = [], []
    t0 = time.perf_counter()
    for c in range(cycles):
        ctx.advance(nx)
        ctx.exchange()
        if (c + 1) % sample == 0:
            H.append(ctx.energies()[2])
            t.append((c + 1) * nx * dt)
    att, acc = ctx.accept_stats()
    return ((acc - acc0) / np.maximum(att - att0, 1)).tolist(), (att - att0).tolist(), \
        drift_slopes(t, H, N), time.perf_counter() - t0


def run_precision(args):
    """Precision study (the 256 x 4000 workload's precision configuration):
    energy drift of H~ per atom per tau over equal-length runs for the mixed
    batched, FP64 batched and plain FP64 paths, and exchange acceptance per
    ladder pair for the two batched paths.  The oracle's legs run on the host
    (tests/precision_oracle.py, the oracle being test infrastructure)."""
    import torch
    import paper_0812_1633_gb300 as re
    from paper_0812_1633_gb300 import build
    build.build()
    N, R, S = PREC_N, PREC_R, args.prec_steps
    L = inputs.box_length(N)
    temps = precision_temps()
    if args.prec_full:
        # the whole 256-replica ladder on the mixed batched path
        full = inputs.geometric_ladder(0.75, 1.8, 256)
        out = {"study": "precision, whole ladder: mixed batched path",
               "workload": f"256 x {N}, T 0.75-1.8 geometric, rho 0.8442, dt 0.005, tau_T 0.5, "
                           f"skin 0.5, FCC start, seed {PREC_SEED}", "steps": S}
        ctx = re.Context(N, L, 2.5, full, PREC_SEED)
        sl, wall = drift_run(ctx, S, 100, N)
        ctx.close()
        out["drift"] = {"slopes": sl.tolist(), "mean": float(np.mean(sl)),
                        "sd": float(np.std(sl, ddof=1)), "max_abs": float(np.abs(sl).max()),
                        "replica_atom_steps_per_s": 256 * N * S / wall}
        print(json.dumps({"drift": out["drift"]}), flush=True)
        ctx = re.Context(N, L, 2.5, full, PREC_SEED)
        acc, att, sl, wall = exchange_run(ctx, S // 10, 10, N)
        ctx.close()
        out["exchange"] = {"nx": 10, "acceptance_per_pair": acc, "attempts_per_pair": att,
                           "slopes": sl.tolist(), "mean_slope": float(np.mean(sl)),
                           "wall_s": wall}
        print(json.dumps(out), flush=True)
        return
    out = {"study": "precision: energy drift and exchange acceptance per path",
           "workload": f"{R} consecutive replicas (the coldest) of the 256-replica ladder T "
                       f"0.75-1.8, N {N}, rho 0.8442, dt 0.005, tau_T 0.5, skin 0.5, FCC start, "
                       f"seed {PREC_SEED}",
           "drift": {"steps": S, "unit": "H~ slope per atom per tau (least squares)"},
           "exchange": {"steps": S, "nx": 10}}
    ends = np.zeros(R, np.int32)
    ends[[0, R - 1]] = 1
    for name, kw in [("mixed_batched", dict(precision="mixed")),
                     ("fp64_batched", dict(precision="fp64")),
                     ("plain_fp64", dict(path="plain"))]:
        ctx = re.Context(N, L, 2.5, temps, PREC_SEED, **kw)
        if name == "plain_fp64":
            # one replica per launch sequence: the two ends of the ladder only
            sl, wall = drift_run(ctx, S, 100, N, budgets=ends)
            sl = sl[[0, R - 1]]
            reps = [0, R - 1]
        else:
            sl, wall = drift_run(ctx, S, 100, N)
            reps = list(range(R))
        out["drift"][name] = {"replicas": reps, "slopes": sl.tolist(),
                              "mean": float(np.mean(sl)), "max_abs": float(np.abs(sl).max()),
                              "replica_atom_steps_per_s": len(reps) * N * S / wall}
        ctx.close()
        print(json.dumps({name: out["drift"][name]}), flush=True)
    for name, kw in [("mixed_batched", dict(precision="mixed")),
                     ("fp64_batched", dict(precision="fp64"))]:
        ctx = re.Context(N, L, 2.5, temps, PREC_SEED, **kw)
        acc, att, sl, wall = exchange_run(ctx, S // 10, 10, N)
        out["exchange"][name] = {"acceptance_per_pair": acc, "attempts_per_pair": att,
                                 "slopes": sl.tolist(), "mean_slope": float(np.mean(sl)),
                                 "wall_s": wall}
        ctx.close()
        print(json.dumps({name + "_exchange": out["exchange"][name]}), flush=True)
    print(json.dumps(out), flush=True)


def melted_context(re, N, temps, seed, **kw):
    """A liquid on the ladder: melted at T 2.0-2.2 from the FCC start, velocities
    rescaled to the ladder, 200 steps on it."""
    L = inputs.box_length(N)
    temps = np.asarray(temps, dtype=np.float64)
    hot = inputs.geometric_ladder(2.0, 2.2, len(temps))
    m = re.Context(N, L, 2.5, hot, seed, **kw)
    m.advance(2000)
    x, v = m.get_state()
    m.close()
    ctx = re.Context(N, L, 2.5, temps, seed + 1, **kw)
    ctx.set_state(x, v * np.repeat(np.sqrt(temps / hot), N)[:, None])
    ctx.advance(200)
    return ctx


def timed(torch, fn):
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    fn()
    torch.cuda.synchronize()
    return time.perf_counter() - t0


def run_lambda(args):
    """Parallel efficiency lambda (Example section, Scalability): total steps of
    all replicas per wall-clock second with exchanges, divided by the same
    without exchanges, against the number of replicas."""
    import torch
    import paper_0812_1633_gb300 as re
    from paper_0812_1633_gb300 import build
    build.build()
    N, nx, A = args.lam_n, args.lam_nx, args.lam_attempts
    out = {"study": "parallel efficiency lambda vs replicas",
           "workload": f"R replicas x {N} atoms, rho 0.8442, T 0.7-2.5 geometric, skin 0.3, "
                       f"mixed, melted start; N_x {nx}; {A} attempts per measurement",
           "modes": {"no_exchange": "one launch, every replica runs until the master has made "
                                    f"{A}*N_x steps (the lambda denominator)",
                     "sync": "per attempt: one launch of N_x steps per replica, then the "
                             "exchange kernel (CUDA graph)",
                     "master_stop": "per attempt: one launch ended by the rotating master "
                                    "after N_x steps, then the exchange kernel (CUDA graph)",
                     "async": "one launch; exchanges between replicas inside it (rotating "
                              "master, pairwise waits)"},
           "rows": []}
    for R in [int(v) for v in args.lam_rs.split(",")]:
        temps = inputs.geometric_ladder(0.7, 2.5, R)
        ctx = melted_context(re, N, temps, 777, skin=0.3, nx=nx)
        try:
            ctx.run_free(2, nx)
            free_ok = True
        except re.REError as e:
            # the free-running launch needs every replica resident: one CTA per
            # replica (one thread per atom) when the default shape has too
            # many clusters; every mode of the row then runs in that shape
            ctx.close()
            ctx = melted_context(re, N, temps, 777, skin=0.3, nx=nx, cluster=1, atom_threads=1)
            try:
                ctx.run_free(2, nx)
                free_ok = True
            except re.REError:
                free_ok = False
                refused = str(e)
        row = {"R": R, "launch": ctx.config()}
        if not free_ok:
            row["async"] = {"unavailable": refused}
        cnt = lambda: ctx.counters()[0].astype(np.float64)
        # warm-up of every mode (graphs, lazily allocated buffers)
        ctx.advance_async(nx)
        ctx.run(2)
        ctx.run_async(2, nx)
        s0 = cnt()
        t = timed(torch, lambda: ctx.advance_async(A * nx))
        rate0 = (cnt() - s0).sum() / t
        row["no_exchange"] = {"replica_steps_per_s": rate0}
        t = timed(torch, lambda: ctx.run(A))
        r_sync = R * nx * A / t
        row["sync"] = {"replica_steps_per_s": r_sync, "lambda": r_sync / rate0, "mean_nx": nx}
        s0 = cnt()
        t = timed(torch, lambda: ctx.run_async(A, nx))
        d = cnt() - s0
        row["master_stop"] = {"replica_steps_per_s": d.sum() / t, "lambda": d.sum() / t / rate0,
                              "mean_nx": d.sum() / (R * A)}
        if free_ok:
            s0 = cnt()
            t = timed(torch, lambda: ctx.run_free(A, nx))
            d = cnt() - s0
            row["async"] = {"replica_steps_per_s": d.sum() / t, "lambda": d.sum() / t / rate0,
                            "mean_nx": d.sum() / (R * A)}
        att, acc = ctx.accept_stats()
        row["acceptance"] = float(acc.sum() / max(att.sum(), 1))
        out["rows"].append(row)
        print(json.dumps(row), flush=True)
        ctx.close()
    print(json.dumps(out), flush=True)


def run_acceptance(args):
    """Exchange acceptance on the paper's workload (Example section: 4000 atoms,
    rho 0.8442, T_k = 0.7 * 1.0275^k) explained by the model's heat capacity:
    the replicas run without exchanges; the configurational heat capacity per
    atom comes from the potential-energy fluctuations, Var(U) / (N T^2), and
    independently from the slope d<U>/dT over the ladder; the acceptance of each
    neighbouring pair is predicted from the sampled energies alone, the mean of
    min(1, exp((1/T_a - 1/T_b)(U_a - U_b))) over pairs of samples, and compared
    with the acceptance the exchanges then measure."""
    import torch
    import paper_0812_1633_gb300 as re
    from paper_0812_1633_gb300 import build
    build.build()
    N, R = 4000, args.acc_r
    temps = inputs.paper_ladder(R)
    ctx = melted_context(re, N, temps, 4242, skin=0.5)
    for _ in range(40):
        ctx.advance(500)
    S, stride = args.acc_samples, 25
    U = np.zeros((S, R))
    for s in range(S):
        ctx.advance(stride)
        U[s] = ctx.energies()[0]
    mean, var = U.mean(0), U.var(0)
    blocks = U[:S - S % 20].reshape(20, -1, R).mean(1)
    err = blocks.std(0, ddof=1) / np.sqrt(20)
    pred = []
    for k in range(R - 1):
        a = 1.0 / temps[k] - 1.0 / temps[k + 1]
        d = a * (U[:, k][:, None] - U[:, k + 1][None, ::7])
        pred.append(float(np.minimum(1.0, np.exp(np.minimum(d, 0.0))).mean()))
    # then the exchanges themselves
    att0, acc0 = ctx.accept_stats()
    for _ in range(args.acc_attempts):
        ctx.advance(10)
        ctx.exchange()
    att, acc = ctx.accept_stats()
    att, acc = att - att0, acc - acc0
    out = {"study": "exchange acceptance vs heat capacity",
           "workload": f"{R} replicas x {N} atoms, rho 0.8442, T_k = 0.7 * 1.0275^k, skin 0.5, "
                       f"mixed, melted start; {S} samples every {stride} steps without exchanges, "
                       f"then {args.acc_attempts} attempts every 10 steps",
           "T": temps.tolist(), "U_per_atom": (mean / N).tolist(),
           "U_err_per_atom": (err / N).tolist(),
           "C_conf_from_fluctuations": (var / (N * temps ** 2)).tolist(),
           "C_conf_from_slope": float(np.polyfit(temps, mean, 1)[0] / N),
           "acceptance_predicted_per_pair": pred,
           "acceptance_predicted_mean": float(np.mean(pred)),
           "acceptance_measured_per_pair": (acc / np.maximum(att, 1)).tolist(),
           "acceptance_measured_mean": float(acc.sum() / max(att.sum(), 1))}
    ctx.close()
    print(json.dumps(out), flush=True)


def msd_diffusion(logT, steps, max_lag=10):
    """D of ln T: half the slope of the mean squared displacement of ln T against
    elapsed steps, over lags of 1..max_lag attempts (least squares through 0).
    logT, steps: (attempts, replicas)."""
    y = np.log(logT)
    lags, msd = [], []
    for m in range(1, max_lag + 1):
        dy = y[m:] - y[:-m]
        ds = steps[m:] - steps[:-m]
        lags.append(ds.mean())
        msd.append((dy * dy).mean())
    lags, msd = np.asarray(lags), np.asarray(msd)
    return float((lags * msd).sum() / (lags * lags).sum() / 2.0)


def diffusion_sync_trajectory(ctx, nx, attempts):
    """Synchronous scheme: every attempt, each replica advances nx steps and
    the ladder attempts its exchanges.  Returns the temperature of every
    replica after each attempt and the steps it has made since the start
    (both (attempts, replicas))."""
    base = ctx.counters()[0]
    Ts, st = [], []
    for _ in range(attempts):
        ctx.advance(nx)
        ctx.exchange()
        Ts.append(ctx.temps())
        st.append(ctx.counters()[0] - base)
    return np.array(Ts), np.array(st, dtype=np.float64)


def diffusion_async_trajectory(ctx, nx, attempts):
    """Asynchronous scheme (one free-running launch, rotating master after nx
    of its own steps): the log's temperature after each attempt and the step
    at which each replica took part, counted from the start."""
    base = ctx.counters()[0]
    steps, T, _, _ = ctx.run_free(attempts, nx, log=True)
    return T, (steps - base).astype(np.float64)


def run_diffusion(args):
    """Diffusion coefficient of ln T against the observed exchange stride <N_x>
    (Example section, Diffusion in temperature space) for the synchronous and
    the asynchronous (in-launch) schemes."""
    import torch
    import paper_0812_1633_gb300 as re
    from paper_0812_1633_gb300 import build
    build.build()
    N, R, A = args.dif_n, args.dif_r, args.dif_attempts
    ratio = args.dif_ratio
    temps = 0.7 * ratio ** np.arange(R)
    out = {"study": "diffusion coefficient of ln T vs <N_x>",
           "workload": f"{R} replicas x {N} atoms, rho 0.8442, T_k = 0.7 * {ratio}^k, skin 0.3, "
                       f"mixed, melted start, {A} attempts per point, cluster "
                       f"{args.dif_cluster}",
           "estimator": "half the least-squares slope (through 0) of <(ln T(t+s) - ln T(t))^2> "
                        "against the elapsed steps s, lags of 1-10 attempts",
           "rows": []}
    for nx in [int(v) for v in args.dif_nx.split(",")]:
        row = {"nx": nx}
        # one launch shape for both schemes, with every replica resident
        shape = dict(skin=0.3, nx=nx, cluster=args.dif_cluster, atom_threads=1)
        ctx = melted_context(re, N, temps, 4242, **shape)
        Ts, st = diffusion_sync_trajectory(ctx, nx, A)
        att, acc = ctx.accept_stats()
        row["sync"] = {"D": msd_diffusion(Ts, st), "mean_nx": nx,
                       "acceptance": float(acc.sum() / att.sum())}
        ctx.close()
        ctx = melted_context(re, N, temps, 4242, **shape)
        try:
            a0, c0 = ctx.accept_stats()
            T, steps = diffusion_async_trajectory(ctx, nx, A)
            att, acc = ctx.accept_stats()
            mean_nx = float(np.diff(np.vstack([np.zeros((1, R)), steps]), axis=0).mean())
            row["async"] = {"D": msd_diffusion(T, steps), "mean_nx": mean_nx,
                            "acceptance": float((acc - c0).sum() / (att - a0).sum())}
        except re.REError as e:
            row["async"] = {"unavailable": str(e)}
        ctx.close()
        out["rows"].append(row)
        print(json.dumps(row), flush=True)
    print(json.dumps(out), flush=True)


# DRAM bytes (read + write) per launch of the advance kernel, from one ncu
# capture per workload and launch shape (its summary is in profiles/),
# valid only while the kernel's sources are the ones that were profiled.
PROFILED_TRAFFIC = {
    ("c1", (2, 2, 2), "mixed"): {"kernel_sha256_16": "9b8dd646a6bec915",
                                 "bytes_per_launch": 14288896 + 69376,
                                 # pipe use over the SMs' active cycles (ncu --set full)
                                 "pipes": {"fma_pct": 19.94, "alu_pct": 40.73, "fp64_pct": 4.46,
                                           "issue_active_pct": 53.41,
                                           "smem_wavefronts": 18227323,
                                           "smem_bank_conflicts": 7456171}},
}


def kernel_sources_hash():
    import hashlib
    h = hashlib.sha256()
    here = os.path.join(os.path.dirname(os.path.abspath(__file__)), "paper_0812_1633_gb300",
                        "csrc")
    for f in ("re_md.cuh", "re_batched.cuh", "re_batched_mix.cu", "re_batched_mix_narrow.cu",
              "re_device.cuh", "re_internal.h"):
        with open(os.path.join(here, f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def profiled_record(config, launch, prec):
    """The ncu capture of this workload's launch shape, or None when the kernel
    changed since the capture (or this shape was not captured)."""
    key = (config, (launch.get("cluster"), launch.get("atom_threads"), launch.get("cell_div")),
           prec)
    rec = PROFILED_TRAFFIC.get(key)
    if rec is None or rec["kernel_sha256_16"] != kernel_sources_hash():
        return None
    return rec


def profiled_traffic(config, launch, prec):
    """ncu DRAM traffic per launch for this workload, or None (see profiled_record)."""
    rec = profiled_record(config, launch, prec)
    return None if rec is None else rec["bytes_per_launch"]


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=2000)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--equil-steps", type=int, default=1000,
                    help="untimed MD steps from the FCC start before tuning and timing")
    ap.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    ap.add_argument("--config", default="c1", choices=sorted(CONFIGS))
    ap.add_argument("--cpu-seconds", type=float, default=10.0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-plain", action="store_true", help="skip the plain FP64 comparison")
    ap.add_argument("--graph-cycles", type=int, default=20,
                    help="cycles of the CUDA-graph replay measurement (0: skip)")
    ap.add_argument("--free-attempts", type=int, default=200,
                    help="exchange attempts of the free-running measurement (0: skip)")
    ap.add_argument("--study", default=None,
                    choices=["drift", "lambda", "diffusion", "acceptance", "precision"],
                    help="run a study instead of the throughput bench")
    ap.add_argument("--lam-n", type=int, default=864)
    ap.add_argument("--lam-nx", type=int, default=5)
    ap.add_argument("--lam-attempts", type=int, default=400)
    ap.add_argument("--lam-rs", default="8,16,32,64,96,128,152")
    ap.add_argument("--dif-n", type=int, default=2048)
    ap.add_argument("--dif-r", type=int, default=48)
    ap.add_argument("--dif-ratio", type=float, default=1.0386)
    ap.add_argument("--dif-attempts", type=int, default=2000)
    ap.add_argument("--dif-nx", default="1,2,5,10,20")
    ap.add_argument("--dif-cluster", type=int, default=2)
    ap.add_argument("--acc-r", type=int, default=8)
    ap.add_argument("--acc-samples", type=int, default=4000)
    ap.add_argument("--acc-attempts", type=int, default=2000)
    ap.add_argument("--prec-steps", type=int, default=100000)
    ap.add_argument("--prec-full", action="store_true",
                    help="precision study: the whole 256-replica ladder, mixed path only")
    ap.add_argument("--drift-n", type=int, default=4000)
    ap.add_argument("--drift-r", type=int, default=8)
    ap.add_argument("--drift-steps", type=int, default=20000)
    ap.add_argument("--drift-window", type=int, default=4000)
    ap.add_argument("--wide", type=int, default=0,
                    help="with --launch: split launch 1 (where it applies), -1 never, 0 default")
    ap.add_argument("--launch", default=None,
                    help="fixed launch shape 'cluster,atom_threads,cell_div' instead of the autotuner")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    cfg = CONFIGS[args.config]
    if args.study == "drift":
        run_drift(args)
        return
    if args.study == "lambda":
        run_lambda(args)
        return
    if args.study == "diffusion":
        run_diffusion(args)
        return
    if args.study == "acceptance":
        run_acceptance(args)
        return
    if args.study == "precision":
        run_precision(args)
        return
    if args.impl == "reference":
        run_reference(args, cfg)
    else:
        run_gpu(args, cfg)


if __name__ == "__main__":
    main()
