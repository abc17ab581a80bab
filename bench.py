#!/usr/bin/env python
"""Throughput benchmark of the on-the-fly RNG + Langevin-dynamics hot path.

One bench step is one pass of the whole hot path over the throughput
workload (10^6 independent 3-D oscillators, the paper's Sec. IV test shape):
  - fused Langevin dynamics, 10^4 steps, for each generator (Hybrid Taus,
    Ran2, Lagged Fibonacci on the last Table I row), seeding excluded;
  - stand-alone fills of 2^30 uniform and 2^30 normal binary32 numbers per
    generator;
  - 512 uneven systems (N log-uniform in [1e2, 1e5]) x 5000 steps in one
    batched graph launch, and the adjoint of 1e5 oscillators x 1e4 steps for
    Hybrid Taus and Ran2 (noise regenerated from checkpoints every 100 steps).
value = oscillator-steps advanced per second over the whole step (fills
count toward the time, not the oscillator-steps).  Inputs stay resident in
HBM; the L2 (126 MB) is flushed by a 256 MiB write before every timed part.
After the timed steps, the large workload (10^8 oscillators x 1000 steps per
generator) is timed once per generator, outside the step, and reported per
part with its roofline.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl gbrng|reference]

With --impl reference the CPU oracle is timed on bounded samples of the same
workload on this machine's host cores (oracle/ is test infrastructure; only
that leg and the cpu_baseline leg run it).
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
sys.path.insert(0, ROOT)

from paper_1003_1123_gb300 import workloads as W  # noqa: E402  (seeded inputs only)

N_OSC = 10**6
LD_STEPS = 10**4
FILL_N = 2**30
SEED = 2024
KINDS = ("taus", "ran2", "lagfib")
L2_FLUSH_BYTES = 256 << 20
PARAMS = dict(K=1.0, m=1.0, gamma=0.5, kT=1.0, dt=0.01)
BATCH_SYSTEMS, BATCH_STEPS = 512, 5000
ADJ_N, ADJ_STEPS, ADJ_CKPT = 10**5, 10**4, 100
ADJ_KINDS = ("taus", "ran2")
LARGE_N, LARGE_STEPS = 10**8, 1000
LARGE_PARAMS = dict(K=1.0, m=1.0, gamma=1.0, kT=1.0, dt=0.01)
STEPWISE_STEPS = 1000
WORKLOAD = ("N=1e6 3-D oscillators x 1e4 fused steps per generator (Taus, Ran2, Lagged "
            "Fibonacci row 9) + 2^30 uniform and 2^30 normal fills per generator + 512 uneven "
            "systems (N 1e2..1e5) x 5000 batched steps + adjoint (Taus, Ran2) of 1e5 "
            "oscillators x 1e4 steps")

# Integer-ALU-pipe instructions a draw needs as the algorithm is printed, given the
# instruction set (LOP3 evaluates any three-input logic function, SHF is one shift, and
# left shifts, multiplies and adds can run as IMAD on the FMA pipe instead):
#   Hybrid Taus, per Tausworthe word ((y << s1) ^ y) >> s2, ((y & c) << s3) ^ b:
#     the xor (LOP3), the right shift (SHF) and the masked xor (LOP3) = 3, the
#     two left shifts on IMAD; 3 words = 9, the LCG word one IMAD (FMA pipe),
#     the four-way xor 2 LOP3 -> 11 per draw, 44 per oscillator-step;
#   Ran2, per a*x mod m from the 64-bit product (IMAD.WIDE on the FMA pipe):
#     the 31-bit funnel shift of the product (SHF), the low-bit mask (LOP3) and
#     the conditional subtraction as an unsigned min of r and r - m (IMNMX) = 3,
#     two of them 6; the slot index iy / NDIV (multiply-high on IMAD, one SHF)
#     1; the wrap of iy as min_u32(y, y + m1 - 1) 1 -> 8 per draw, 32 per
#     oscillator-step.
# A fixed yardstick for the 64-lane ALU pipe.  The Hybrid Taus kernels need fewer since
# they step the words by funnel shifts (29 an oscillator-step), so for them it is a rate
# in the printed algorithm's operations and no lower bound; ncu's measured ALU-pipe
# utilisation is reported beside it.
INT_OPS_PER_DRAW = {"taus": 11, "ran2": 8}
INT_OPS_PER_OSC_STEP = {k: 4 * v for k, v in INT_OPS_PER_DRAW.items()}
# Algorithmic bytes per oscillator-step of the Lagged Fibonacci fused step at
# 1e6 oscillators: four ring values, each 2 lag reads + 1 write of 4 B = 48 B
# (x and v stay in shared memory for the whole launch).  The ring (40 MB for
# the last Table I row) stays in L2, so the bound is L2 bandwidth, measured
# below as a device-to-device copy of 2 x 32 MiB that stays L2-resident.
LFG_BYTES_PER_OSC_STEP = 48
# At 1e8 oscillators x and v no longer fit on chip: every step reads and
# writes them (6 binary32 each way), 48 B per oscillator-step of HBM traffic.
LFG_XV_BYTES_PER_OSC_STEP = 48
L2_COPY_BYTES = 32 << 20
FILL_BYTES_PER_NUMBER = 4
# A Lagged Fibonacci fill number as the recurrence is printed: 2 lag reads + 1 ring
# write + 1 output write of 4 B, all through L2 (the ring stays there; the output streams
# on to HBM).  The fans read 1.5 words a number instead of 2, and L2 serves more than a
# copy's bandwidth, so the fraction of the copy can pass 1.
LFG_FILL_BYTES_PER_NUMBER = 16
# DRAM bytes (read + written) of one launch of a part's kernel from the ncu
# capture summarised in profiles/ (same kernel, same launch shape), keyed by
# part and the batched tuner's (T, K, steps per launch); reported as the
# roofline's `traffic` only when this run chose that shape.
NCU_TRAFFIC = {("batched_taus", (64, 2, 0)): 302.788864e6 + 237.262336e6}
# ncu's ALU-pipe utilisation (sm__pipe_alu_cycles_active, % of peak sustained
# active) of each ALU-bound part's kernel, from the captures summarised in
# profiles/alu_pipe_by_part.md (same kernel and launch shape as the bench;
# 100 steps of the 1e6-oscillator systems, 1000 steps of the adjoint, 2^28
# fill numbers, the batched graph's replay; the large parts at 1e7
# oscillators x 10 steps).
NCU_ALU_PIPE_PCT = {"ld_taus": 59.4, "batched_taus": 59.9, "ld_ran2": 51.3,
                    "adjoint_taus": 52.4, "adjoint_ran2": 46.4,
                    "fill_uniform_taus": 82.6, "fill_normal_taus": 70.4,
                    "fill_uniform_ran2": 73.2, "fill_normal_ran2": 56.6,
                    "ld_taus_1e8": 42.9, "ld_ran2_1e8": 39.3}


def load_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            return json.load(f), "measured"
    return {"hbm_gbs": 6800.0, "sm_max_mhz": 2070.0}, "fallback"


# Peak integer-ALU rate: 152 SMs x 64 INT32 lanes per SM (four partitions of 16)
# x SM clock.  The lane count was measured with an issue-rate microbenchmark on
# this GPU (LOP3/SHF 62-69 ops per clock per SM, IMAD 62, MUFU 32); the clock is
# the median sampled during the timed region.
SMS = 152
INT32_LANES_PER_SM = 64


class Clocks:
    """nvidia-smi sampling of SM clocks and throttle reasons during timing."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device_index: int):
        self.dev = device_index
        self.proc = None
        self.path = None

    def start(self):
        fd, self.path = tempfile.mkstemp(prefix="clocks", suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.dev), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except (OSError, FileNotFoundError):
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        rows = []
        with open(self.path) as f:
            for line in f:
                parts = [p.strip() for p in line.split(",")]
                if len(parts) >= 9 and parts[1].isdigit():
                    rows.append(parts)
        os.unlink(self.path)
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        mhz = [int(r[1]) for r in rows]
        reasons = set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in rows:
            for name, val in zip(names, r[5:9]):
                if val.lower().startswith("active"):
                    reasons.add(name)
        return {"sm_mhz": statistics.median(mhz), "sm_max_mhz": int(rows[0][2]),
                "power_w_max": max(float(r[3]) for r in rows if r[3].replace(".", "").isdigit())
                if any(r[3].replace(".", "").isdigit() for r in rows) else None,
                "samples": len(rows), "reasons": sorted(reasons)}


# ------------------------------------------------------------- replicas
def rank_seed(rank: int) -> int:
    """Seed of a rank's replica: independent streams per rank (counter-based
    seeding, so ranks share no stream)."""
    return SEED + 1000003 * rank


def max_over_ranks(value: float, dist, device: str) -> float:
    """The slowest rank's time: one all-reduce (MAX) of a scalar, the only
    collective of a replicas run."""
    if not dist:
        return value
    import torch
    t = torch.tensor([value], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_rate(world: int, units_per_step: float, ms_per_step: float) -> float:
    """Units all ranks processed per second (each rank runs the full step)."""
    return world * units_per_step / (ms_per_step / 1e3)


# --------------------------------------------------------------------- GPU
class Workload:
    def __init__(self, G, torch, rank: int):
        self.G, self.torch = G, torch
        seed = rank_seed(rank)
        self.systems = {}
        for kind in KINDS:
            r = G.rng_init(kind, seed, N_OSC)
            x = torch.zeros((N_OSC, 3), dtype=torch.float32, device="cuda")
            v = torch.zeros_like(x)
            s = G.LdSystem(r, x, v, **PARAMS)
            G.ld_init_equilibrium(s)
            self.systems[kind] = s
        self.fill_rngs = {k: G.rng_init(k, seed + 7, N_OSC) for k in KINDS}
        self.out = torch.empty(FILL_N, dtype=torch.float32, device="cuda")
        self.flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.float32, device="cuda")
        # batched: 512 uneven systems (Hybrid Taus), one graph launch per call;
        # their x, v are consecutive slices of two arrays, so a host round trip
        # of the whole batch is one copy each way
        specs = W.batched_systems(BATCH_SYSTEMS, seed=1234 + rank)
        self.batch_osc = sum(sp["n"] for sp in specs)
        self.batch_x = torch.zeros((self.batch_osc, 3), dtype=torch.float32, device="cuda")
        self.batch_v = torch.zeros_like(self.batch_x)
        self.batch = []
        off = 0
        for sp in specs:
            r = G.rng_init("taus", sp["seed"], sp["n"])
            n = sp["n"]
            s = G.LdSystem(r, self.batch_x[off:off + n], self.batch_v[off:off + n], K=sp["K"],
                           m=sp["m"], gamma=sp["gamma"], kT=sp["kT"], dt=sp["dt"])
            G.ld_init_equilibrium(s)
            self.batch.append(s)
            off += n
        # adjoint: 1e5 oscillators, K per oscillator, checkpoints every 100
        # steps, one system per generator
        self.adj = {}
        for j, kind in enumerate(ADJ_KINDS):
            ra = G.rng_init(kind, seed + 11 + j, ADJ_N)
            xa = torch.zeros((ADJ_N, 3), dtype=torch.float32, device="cuda")
            sa = G.LdSystem(ra, xa, torch.zeros_like(xa), K_per=torch.ones(ADJ_N, device="cuda"),
                            **{k: v for k, v in PARAMS.items() if k != "K"})
            G.ld_init_equilibrium(sa)
            self.adj[kind] = sa
        self.dK = torch.empty(ADJ_N, dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()

    def parts(self):
        G = self.G
        out = []
        for kind in KINDS:
            s = self.systems[kind]
            out.append((f"ld_{kind}", N_OSC * LD_STEPS, lambda s=s: G.ld_run(s, LD_STEPS)))
        for kind in KINDS:
            r = self.fill_rngs[kind]
            out.append((f"fill_uniform_{kind}", 0,
                        lambda r=r: G.rng_fill_uniform(r, FILL_N, out=self.out)))
            out.append((f"fill_normal_{kind}", 0,
                        lambda r=r: G.rng_fill_normal(r, FILL_N, out=self.out)))
        out.append(("batched_taus", self.batch_osc * BATCH_STEPS,
                    lambda: G.ld_run_batched(self.batch, BATCH_STEPS)))
        for kind in ADJ_KINDS:
            out.append((f"adjoint_{kind}", ADJ_N * ADJ_STEPS,
                        lambda s=self.adj[kind]: adjoint_regenerating(G, s, self.dK)))
        return out

    def step(self, parts, events):
        for i, (_, _, fn) in enumerate(parts):
            self.flush.fill_(float(i))
            events[i][0].record()
            fn()
            events[i][1].record()


def adjoint_regenerating(G, s, dK):
    """ld_backward with the noise regenerated from the checkpointed generator
    states (history limit 0), the adjoint's memory-lean form."""
    G.ld_set_adjoint_history_limit(0)
    try:
        return G.ld_backward(s, ADJ_STEPS, ADJ_CKPT, dK=dK)
    finally:
        G.ld_set_adjoint_history_limit(-1)


def run_gpu(args, rank, world, dist):
    import torch
    from paper_1003_1123_gb300 import gbrng as G

    dev = int(os.environ.get("LOCAL_RANK", 0))
    torch.cuda.set_device(dev)
    wl = Workload(G, torch, rank)
    parts = wl.parts()
    osc_steps_per_step = sum(p[1] for p in parts)
    ev = [[torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)]
          for _ in parts]
    for _ in range(args.warmup):
        wl.step(parts, ev)
    torch.cuda.synchronize()

    part_ms = {name: 0.0 for name, _, _ in parts}
    clocks = Clocks(dev)
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    clocks.start()
    t_start = torch.cuda.Event(enable_timing=True)
    t_end = torch.cuda.Event(enable_timing=True)
    t_start.record()
    for _ in range(args.steps):
        wl.step(parts, ev)
        torch.cuda.synchronize()
        for i, (name, _, _) in enumerate(parts):
            part_ms[name] += ev[i][0].elapsed_time(ev[i][1])
    t_end.record()
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    clk = clocks.stop()
    elapsed_ms = max_over_ranks(t_start.elapsed_time(t_end), dist, "cuda")
    ms_per_step = elapsed_ms / args.steps
    value = whole_job_rate(world, osc_steps_per_step, ms_per_step)

    # ---- end to end through host buffers (pinned inputs and outputs)
    e2e = run_e2e(args, wl, parts, G, torch)

    # ---- roofline of the dominant part, and of every part
    peaks, peak_src = load_peaks()
    dom = max(part_ms, key=part_ms.get)
    dom_ms = part_ms[dom] / args.steps
    units_of = {name: units for name, units, _ in parts}
    l2_gbs = measure_l2_copy_gbs(torch)
    roof = roofline(dom, dom_ms, units_of[dom], peaks, peak_src, clk, l2_gbs)
    roof["traffic"] = NCU_TRAFFIC.get((dom, tuple(G.ld_batched_tune(wl.batch))))
    if roof["traffic"] is not None:
        roof["traffic_source"] = ("ncu dram__bytes_read.sum + dram__bytes_write.sum, one launch of "
                                  "the same kernel and launch shape (committed batched-kernel "
                                  "profile summary)")
    per_part = {name: {"ms": round(part_ms[name] / args.steps, 4)} for name in part_ms}
    for name in part_ms:
        r = roofline(name, part_ms[name] / args.steps, units_of[name], peaks, peak_src, clk, l2_gbs)
        per_part[name]["roofline"] = {k: r[k] for k in ("bound", "achieved", "unit", "frac", "alt",
                                                         "ncu_alu_pipe_pct") if k in r}
    for name, units, _ in parts:
        if units:
            per_part[name]["osc_steps_per_s"] = units / (part_ms[name] / args.steps / 1e3)
        else:
            per_part[name]["numbers_per_s"] = FILL_N / (part_ms[name] / args.steps / 1e3)
            per_part[name]["GBps"] = FILL_N * 4 / (part_ms[name] / args.steps / 1e3) / 1e9
    extras = compare_paths(wl, G, torch, part_ms, args.steps)

    # ---- the large workload, outside the step: 1e8 oscillators x 1000 steps
    del wl
    torch.cuda.empty_cache()
    large, large_clk = run_large(G, torch, dev, peaks, peak_src, l2_gbs)
    per_part.update(large)

    line = {
        "metric": "oscillator-steps/s (fused LD+RNG, all generators, whole hot path)",
        "value": value,
        "unit": "oscillator-steps/s",
        "n_gpus": world,
        "steps": args.steps,
        "warmup": args.warmup,
        "ms_per_step": ms_per_step,
        "higher_is_better": True,
        "scaling": "weak",
        "vs_baseline": None,
        "dtype": "f32+u32",
        "data": "synthetic (seeded oscillators; equilibrium start)",
        "config": bench_config(world, extras["batched_osc"]),
        "clocks": clk,
        "gpu_launches": gpu_launches(parts, args.steps, extras["batched_tune"])
        - in_kernel_statistics(parts) * args.steps,
        "batched_tune": extras["batched_tune"],
        "e2e": e2e,
        "roofline": roof,
        "parts": per_part,
        "comparisons": extras,
        "large_clocks": large_clk,
    }
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(parts, part_ms, args.steps)
    # per-generator headline figures as flat keys of the roofline record (the
    # metric is quoted per generator), repeated as the line's last key
    head = headline(per_part)
    roof.update(head)
    line["per_generator"] = head
    return line


def bench_config(world, batched_osc):
    """The workload's description, the same for both arms."""
    return {"workload": WORKLOAD,
            "batched": {"systems": BATCH_SYSTEMS, "oscillators": batched_osc, "steps": BATCH_STEPS},
            "adjoint": {"n": ADJ_N, "steps": ADJ_STEPS, "checkpoint_every": ADJ_CKPT,
                        "noise": "regenerated from checkpoints"},
            "large": {"n": LARGE_N, "steps": LARGE_STEPS, "params": LARGE_PARAMS,
                      "timed": "once per generator after the steps, outside the step"},
            "n_oscillators": N_OSC, "ld_steps": LD_STEPS, "fill_numbers": FILL_N,
            "params": PARAMS, "l2": "flushed (256 MiB write) before every part",
            "parallelism": f"replicas x{world} (independent seeds, no collective)"}


def headline(per_part):
    """Per-generator fused rates and roofline fractions: the throughput
    workload (1e6 oscillators), the large one (1e8), the adjoint."""
    out = {}
    for name, rec in per_part.items():
        if not (name.startswith("ld_") or name.startswith("adjoint_")):
            continue
        out[f"{name}.osc_steps_per_s"] = rec.get("osc_steps_per_s")
        r = rec.get("roofline", {})
        out[f"{name}.frac"] = r.get("frac")
        out[f"{name}.bound"] = r.get("bound")
        if "ncu_alu_pipe_pct" in r:
            out[f"{name}.ncu_alu_pipe_pct"] = r["ncu_alu_pipe_pct"]
    return out


def run_large(G, torch, dev, peaks, peak_src, l2_gbs):
    """The large workload: 1e8 independent 3-D oscillators x 1000 steps per
    generator (x, v 2.4 GB; Ran2 state 14 GB), K = gamma = kT = 1, dt = 0.01,
    one system at a time.  A 100-step warm-up run, then one timed 1000-step
    run (CUDA events on the launching stream, L2 flushed before it)."""
    flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.float32, device="cuda")
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    clocks = Clocks(dev)
    out = {}
    clocks.start()
    for kind in KINDS:
        r = G.rng_init(kind, SEED + 5, LARGE_N)
        x = torch.zeros((LARGE_N, 3), dtype=torch.float32, device="cuda")
        v = torch.zeros_like(x)
        s = G.LdSystem(r, x, v, **LARGE_PARAMS)
        G.ld_init_equilibrium(s)
        G.ld_run(s, 100, stats=False)
        flush.fill_(1.0)
        a.record()
        G.ld_run(s, LARGE_STEPS)
        b.record()
        torch.cuda.synchronize()
        ms = a.elapsed_time(b)
        name = f"ld_{kind}_1e8"
        units = LARGE_N * LARGE_STEPS
        rf = roofline(name, ms, units, peaks, peak_src, {"sm_mhz": None}, l2_gbs)
        out[name] = {"ms": round(ms, 3), "osc_steps_per_s": units / (ms / 1e3),
                     "outside_step": True,
                     "roofline": {k: rf[k] for k in ("bound", "achieved", "unit", "frac", "alt",
                                                     "ncu_alu_pipe_pct") if k in rf}}
        del s, x, v, r
        torch.cuda.empty_cache()
    clk = clocks.stop()
    # fractions against the clock seen during these runs
    for name, rec in out.items():
        rf = roofline(name, rec["ms"], LARGE_N * LARGE_STEPS, peaks, peak_src, clk, l2_gbs)
        rec["roofline"] = {k: rf[k] for k in ("bound", "achieved", "unit", "frac", "alt",
                                              "ncu_alu_pipe_pct") if k in rf}
    return out, clk


def gpu_launches(parts, steps, batched_tune=None):
    """Kernels of ours launched per timed step: one persistent kernel per fused
    run plus the statistics finisher, one kernel per fill, and for the batched
    graph ceil(steps / L) persistent launches plus the per-system reduction."""
    n = 0
    for name, _, _ in parts:
        if name.startswith("ld_") or name.startswith("adjoint"):
            n += 2                  # persistent kernel + statistics finisher
        elif name.startswith("batched"):
            L = batched_tune[2] if batched_tune else 0
            n += (-(-BATCH_STEPS // L) if L > 0 else 1) + 1
        else:
            n += 1
    return n * steps


def in_kernel_statistics(parts):
    """Runs whose last block adds the statistics up, with no finisher of their own: the
    Lagged Fibonacci run, of one block an SM."""
    return sum(name.startswith("ld_lagfib") for name, _, _ in parts)


def compare_paths(wl, G, torch, part_ms, steps):
    """Outside the timed region: the batched systems run one ld_run each (the
    per-system alternative the batched graph replaces); per adjoint system a
    plain forward run (the adjoint's cost relative to a forward) and the
    adjoint keeping the forward run's noise instead of regenerating it; the
    paper form (one launch per step) on the throughput systems."""
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)

    def timed(fn):
        torch.cuda.synchronize()
        a.record()
        fn()
        b.record()
        torch.cuda.synchronize()
        return a.elapsed_time(b)

    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for s in wl.batch:
        G.ld_run(s, BATCH_STEPS, stats=False)
    torch.cuda.synchronize()
    per_system_ms = 1e3 * (time.perf_counter() - t0)
    batched_ms = part_ms["batched_taus"] / steps
    out = {"batched_ms": batched_ms, "per_system_launches_ms": per_system_ms,
           "batched_speedup": per_system_ms / batched_ms, "batched_osc": wl.batch_osc,
           "batched_tune": list(G.ld_batched_tune(wl.batch))}
    for kind, sa in wl.adj.items():
        fwd_ms = timed(lambda: G.ld_run(sa, ADJ_STEPS))
        adj_ms = part_ms[f"adjoint_{kind}"] / steps
        G.ld_backward(sa, ADJ_STEPS, ADJ_CKPT, dK=wl.dK)      # sizes the history scratch
        hist_ms = timed(lambda: G.ld_backward(sa, ADJ_STEPS, ADJ_CKPT, dK=wl.dK))
        out[f"adjoint_{kind}"] = {
            "regenerating_ms": adj_ms, "forward_ms": fwd_ms,
            "regenerating_over_forward": adj_ms / fwd_ms,
            "with_noise_history_ms": hist_ms, "with_noise_history_over_forward": hist_ms / fwd_ms}
    # the paper form (one launch per step, state through global memory) on the
    # same 1e6-oscillator systems, STEPWISE_STEPS steps, per step vs persistent
    for kind, sysm in wl.systems.items():
        sw = timed(lambda: G.ld_run_stepwise(sysm, STEPWISE_STEPS, stats=False)) / STEPWISE_STEPS
        pers = part_ms[f"ld_{kind}"] / steps / LD_STEPS
        out[f"stepwise_{kind}_us_per_step"] = 1e3 * sw
        out[f"persistent_{kind}_us_per_step"] = 1e3 * pers
        out[f"persistent_speedup_{kind}"] = sw / pers
    return out


def run_e2e(args, wl, parts, G, torch):
    """The same step with inputs in pinned host memory: x, v of every fused
    system copied host->device before and device->host after its run (plus
    its statistics); each fill's first 4 KiB read back to the host.  Every
    part's device buffers are its own, so each step issues all the inputs on
    a copy stream at once, each part waits only for its own, and its results
    go back on a second copy stream while the later parts compute; the step
    ends when every copy has landed."""
    host = {}
    for kind, s in wl.systems.items():
        host[kind] = (s.x.cpu().pin_memory(), s.v.cpu().pin_memory())
    host_batch = (wl.batch_x.cpu().pin_memory(), wl.batch_v.cpu().pin_memory())
    host_adj = {k: (sa.x.cpu().pin_memory(), sa.v.cpu().pin_memory(),
                    torch.empty(ADJ_N, dtype=torch.float32).pin_memory())
                for k, sa in wl.adj.items()}
    probe = torch.empty(1024, dtype=torch.float32).pin_memory()
    main = torch.cuda.current_stream()
    s_in, s_out = torch.cuda.Stream(), torch.cuda.Stream()

    def inputs(name):
        """(device, pinned host) pairs a part reads."""
        if name.startswith("batched"):
            return [(wl.batch_x, host_batch[0]), (wl.batch_v, host_batch[1])]
        if name.startswith("adjoint"):
            k = name.split("_")[-1]
            return [(wl.adj[k].x, host_adj[k][0]), (wl.adj[k].v, host_adj[k][1])]
        if name.startswith("ld_"):
            s = wl.systems[name[3:]]
            return [(s.x, host[name[3:]][0]), (s.v, host[name[3:]][1])]
        return []

    def outputs(name):
        """(pinned host, device) pairs a part's results go to, and the bytes
        of host-side statistics its call returns."""
        if name.startswith("batched"):
            return [(host_batch[0], wl.batch_x), (host_batch[1], wl.batch_v)], 40 * len(wl.batch)
        if name.startswith("adjoint"):
            return [(host_adj[name.split("_")[-1]][2], wl.dK)], 24
        if name.startswith("ld_"):
            s = wl.systems[name[3:]]
            return [(host[name[3:]][0], s.x), (host[name[3:]][1], s.v)], 40
        return [(probe, wl.out[:1024])], 0

    h2d = d2h = 0
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        h2d = d2h = 0
        ready = {}
        with torch.cuda.stream(s_in):
            for name, _, _ in parts:
                for dev, hst in inputs(name):
                    dev.copy_(hst, non_blocking=True)
                    h2d += hst.numel() * 4
                ready[name] = torch.cuda.Event()
                ready[name].record(s_in)
        for name, _, fn in parts:
            main.wait_event(ready[name])
            fn()
            done = torch.cuda.Event()
            done.record(main)
            s_out.wait_event(done)
            pairs, stat_bytes = outputs(name)
            # the fills share one output buffer: their 4 KiB probe is read on
            # the compute stream, before the next fill overwrites it
            # (so is the adjoints' shared dK buffer)
            with torch.cuda.stream(s_out if name.startswith(("ld_", "batched")) else main):
                for hst, dev in pairs:
                    hst.copy_(dev, non_blocking=True)
                    d2h += hst.numel() * 4
            d2h += stat_bytes
        torch.cuda.synchronize()
    sec = (time.perf_counter() - t0) / args.steps
    osc = sum(p[1] for p in parts)
    return {"value": osc / sec, "unit": "oscillator-steps/s", "h2d_bytes_per_step": h2d,
            "d2h_bytes_per_step": d2h}


def measure_l2_copy_gbs(torch):
    """L2-resident copy bandwidth: src and dst of 32 MiB each, 50 copies after
    warm-up, bytes read + written over CUDA-event time."""
    src = torch.empty(L2_COPY_BYTES // 4, dtype=torch.float32, device="cuda").fill_(1.0)
    dst = torch.empty_like(src)
    for _ in range(5):
        dst.copy_(src)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record()
    for _ in range(50):
        dst.copy_(src)
    e1.record()
    torch.cuda.synchronize()
    return 2 * L2_COPY_BYTES * 50 / (e0.elapsed_time(e1) / 1e3) / 1e9


def part_kind(part: str) -> str:
    """Generator of a part: the kind name among its underscore-separated words."""
    for k in KINDS:
        if k in part.split("_"):
            return k
    raise ValueError(part)


def roofline(part, ms, units, peaks, src, clk, l2_gbs=None):
    """Roofline of one part against its binding resource.
    - Taus/Ran2 fused, batched and adjoint: the 64-lane integer ALU pipe, with
      the ALU instructions of the generator's printed draws (INT_OPS_PER_DRAW;
      four draws an oscillator-step, drawn twice by the adjoint, whose reverse
      sweep regenerates the noise), and ncu's measured ALU-pipe utilisation
      beside it where a capture exists.
    - Lagged Fibonacci fused at 1e6 oscillators: the L2 copy bandwidth measured
      in this run (48 algorithmic bytes per oscillator-step: four ring values,
      2 lag reads + 1 write each; x and v stay in shared memory).
    - Lagged Fibonacci fused at 1e8: HBM (x and v stream every step: 24 B read
      + 24 B written per oscillator-step), the ring's 48 B in L2 beside it.
    - Taus/Ran2 fills: the HBM copy bandwidth (4 B per number), with the
      minimal ALU work beside it; Lagged Fibonacci fills: L2 (16 B per number),
      with the HBM figure beside it."""
    mhz = clk.get("sm_mhz") or peaks.get("sm_max_mhz", 2070.0)
    kind = part_kind(part)
    sec = ms / 1e3
    alu_peak = SMS * INT32_LANES_PER_SM * mhz * 1e6 / 1e12
    alu_src = f"152 SMs x {INT32_LANES_PER_SM} INT32 lanes x {mhz} MHz (median SM clock under load)"
    ncu = NCU_ALU_PIPE_PCT.get(part)
    if part.startswith("fill_"):
        hbm = FILL_N * FILL_BYTES_PER_NUMBER / sec / 1e9
        r = {"kernel": part, "bound": "hbm", "achieved": hbm, "peak": peaks["hbm_gbs"],
             "unit": "GB/s", "frac": hbm / peaks["hbm_gbs"], "traffic": None,
             "peak_source": f"{src} hbm_gbs (copy bandwidth); 4 B per number"}
        if kind != "lagfib":
            ops = INT_OPS_PER_DRAW[kind] * FILL_N / sec / 1e12
            r["alt"] = {"bound": "alu", "achieved": ops, "unit": "Tops/s", "frac": ops / alu_peak}
            if ncu is not None:
                r["ncu_alu_pipe_pct"] = ncu
            return r
        l2 = FILL_N * LFG_FILL_BYTES_PER_NUMBER / sec / 1e9
        return {"kernel": part, "bound": "l2", "achieved": l2, "peak": l2_gbs, "unit": "GB/s",
                "frac": l2 / l2_gbs if l2_gbs else None, "traffic": None,
                "peak_source": "L2-resident copy of 2 x 32 MiB measured in this run; "
                               "16 B per number",
                "alt": {k: r[k] for k in ("bound", "achieved", "unit", "frac")}}
    if kind == "lagfib":
        l2 = units * LFG_BYTES_PER_OSC_STEP / sec / 1e9
        l2r = {"kernel": part, "bound": "l2", "achieved": l2, "peak": l2_gbs,
               "unit": "GB/s", "frac": l2 / l2_gbs if l2_gbs else None, "traffic": None,
               "peak_source": "L2-resident copy of 2 x 32 MiB measured in this run; "
                              "algorithmic 48 B per oscillator-step (ring)"}
        if not part.endswith("_1e8"):
            return l2r
        hbm = units * LFG_XV_BYTES_PER_OSC_STEP / sec / 1e9
        return {"kernel": part, "bound": "hbm", "achieved": hbm, "peak": peaks["hbm_gbs"],
                "unit": "GB/s", "frac": hbm / peaks["hbm_gbs"], "traffic": None,
                "peak_source": f"{src} hbm_gbs (copy bandwidth); x, v read and written every "
                               "step: 48 B per oscillator-step",
                "alt": {k: l2r[k] for k in ("bound", "achieved", "unit", "frac")}}
    draws = 2 if part.startswith("adjoint_") else 1
    ops = draws * INT_OPS_PER_OSC_STEP[kind] * units
    achieved = ops / sec / 1e12
    r = {"kernel": part, "bound": "alu", "achieved": achieved, "peak": alu_peak,
         "unit": "Tops/s", "frac": achieved / alu_peak, "traffic": None,
         "peak_source": alu_src,
         "ops_source": f"minimal ALU-pipe instructions: {INT_OPS_PER_DRAW[kind]} per draw, "
                       f"{4 * draws} draws per oscillator-step"}
    if ncu is not None:
        r["ncu_alu_pipe_pct"] = ncu
    return r


# --------------------------------------------------------------------- CPU
ORACLE_PARTS = ("ld_taus", "ld_ran2", "ld_lagfib", "fill_uniform_taus", "fill_normal_taus",
                "fill_uniform_ran2", "fill_normal_ran2", "fill_uniform_lagfib",
                "fill_normal_lagfib", "adjoint_taus", "adjoint_ran2")


def _oracle_part(name: str, scale: float, shard: int = 0):
    """One bounded sample of one part on the oracle as it stands, in this
    process; returns (units done, seconds).  Shards of the per-thread kinds use
    disjoint seeds (the oracle's streams are independent)."""
    import numpy as np
    import oracle
    p = oracle.params(**PARAMS)
    seed = SEED + 1009 * shard
    kind = name.split("_")[-1]
    if name.startswith("ld_"):
        if kind == "lagfib":
            g = oracle.Gen(kind, seed, N_OSC)
            x, v = oracle.ld_init_eq_f32(g, N_OSC, p)
            steps = max(1, int(2 * scale))
            t0 = time.perf_counter()
            oracle.ld_run_f32(g, x, v, p, steps)
            return N_OSC * steps, time.perf_counter() - t0
        n, steps = int(20000 * scale), 100
        g = oracle.Gen(kind, seed, n)
        x, v = oracle.ld_init_eq_f32(g, n, p)
        t0 = time.perf_counter()
        oracle.ld_run_f32(g, x, v, p, steps)
        return n * steps, time.perf_counter() - t0
    if name.startswith("fill_"):
        nf = int(2 * 10**6 * scale)
        g = oracle.Gen(kind, seed + 7, N_OSC if kind == "lagfib" else 4096)
        f = g.fill_uniform if "uniform" in name else g.fill_normal
        t0 = time.perf_counter()
        f(nf)
        return nf, time.perf_counter() - t0
    na, sa = max(8, int(200 * scale)), 1000          # adjoint_<kind>, FP64
    g = oracle.Gen(kind, seed + 11, na)
    x, v = oracle.ld_init_eq_f64(g, na, p)
    t0 = time.perf_counter()
    oracle.ld_adjoint_f64(g, x, v, p, sa, Kper=np.ones(na))
    return na * sa, time.perf_counter() - t0


def oracle_pool(workers: int):
    """A process pool for the oracle, started with spawn (no inherited CUDA
    state), or None for one core."""
    if workers <= 1:
        return None
    import concurrent.futures as cf
    import multiprocessing as mp
    return cf.ProcessPoolExecutor(max_workers=workers, mp_context=mp.get_context("spawn"))


def _oracle_rates(budget_scale=1.0, pool=None, workers=1):
    """Time the oracle as it stands on bounded samples of the workload; returns
    per-part rates.  With a pool, each per-thread part runs `workers` shards at
    once and its rate is their units over the wall time; the Lagged Fibonacci
    sequence is serial by definition and stays on one core."""
    rates = {}
    for name in ORACLE_PARTS:
        if pool is None or name.endswith("lagfib"):
            units, sec = _oracle_part(name, budget_scale)
            rates[name] = units / sec
            continue
        t0 = time.perf_counter()
        futs = [pool.submit(_oracle_part, name, budget_scale, k) for k in range(workers)]
        units = sum(f.result()[0] for f in futs)
        rates[name] = units / (time.perf_counter() - t0)
    # batched systems run the same per-oscillator arithmetic as a Taus system
    rates["batched_taus"] = rates["ld_taus"]
    return rates


def _step_units():
    batch_osc = sum(sp["n"] for sp in W.batched_systems(BATCH_SYSTEMS, seed=1234))
    units = {f"ld_{k}": N_OSC * LD_STEPS for k in KINDS}
    units.update({f"fill_{m}_{k}": FILL_N for k in KINDS for m in ("uniform", "normal")})
    units["batched_taus"] = batch_osc * BATCH_STEPS
    for k in ADJ_KINDS:
        units[f"adjoint_{k}"] = ADJ_N * ADJ_STEPS
    return units


def _step_osc_steps(units):
    return sum(u for name, u in units.items() if not name.startswith("fill_"))


def _cpu_step_seconds(rates):
    units = _step_units()
    return sum(units[name] / r for name, r in rates.items())


def _sample_text(scale, workers=1):
    per = f" in each of {workers} concurrent processes (Lagged Fibonacci on one)" if workers > 1 else ""
    return (f"per generator: Taus/Ran2 {int(20000 * scale)} oscillators x 100 steps, Lagged "
            f"Fibonacci all 1e6 oscillators x {max(1, int(2 * scale))} steps, "
            f"{int(2e6 * scale)} uniform + {int(2e6 * scale)} normal fill numbers, "
            f"FP64 adjoint of {max(8, int(200 * scale))} oscillators x 1000 steps{per} (batched "
            f"systems at the Taus rate); extrapolated per unit to the full step")


def host_cpu() -> str:
    """The host's architecture and core model, as the kernel reports it
    (x86 "model name"; Arm implementer and part numbers)."""
    import platform
    model = ""
    try:
        with open("/proc/cpuinfo") as f:
            info = {}
            for line in f:
                if ":" in line:
                    k, v = line.split(":", 1)
                    info.setdefault(k.strip(), v.strip())
        model = info.get("model name") or " ".join(
            f"{k} {info[k]}" for k in ("CPU implementer", "CPU part") if k in info)
    except OSError:
        pass
    return f"{platform.machine()} {model}".strip()


def cpu_baseline(parts, part_ms, steps):
    """The oracle on all host cores (spawned processes over independent
    streams), and on one core for reference."""
    workers = os.cpu_count() or 1
    pool = oracle_pool(workers)
    try:
        rates = _oracle_rates(1.0, pool, workers)
    finally:
        if pool:
            pool.shutdown()
    one = _oracle_rates(1.0)
    units = _step_osc_steps(_step_units())
    return {"value": units / _cpu_step_seconds(rates), "unit": "oscillator-steps/s",
            "cores": workers, "cpu": host_cpu(), "kind": "oracle",
            "sample": _sample_text(1.0, workers),
            "parts": {k: v for k, v in rates.items()},
            "one_core": {"value": units / _cpu_step_seconds(one), "cores": 1,
                         "parts": {k: v for k, v in one.items()}}}


def run_reference(args, world):
    """The oracle on the host cores, timed like our arm: W untimed and K timed
    steps, each a bounded sample of the workload; value is the rate of the
    samples extrapolated per unit to the whole step, ms_per_step the measured
    wall time of a timed (sample) step."""
    scale = 0.5
    workers = os.cpu_count() or 1
    pool = oracle_pool(workers)
    try:
        for _ in range(args.warmup):
            _oracle_rates(0.1, pool, workers)
        secs = []
        t0 = time.perf_counter()
        for _ in range(args.steps):
            secs.append(_cpu_step_seconds(_oracle_rates(scale, pool, workers)))
        wall = time.perf_counter() - t0
    finally:
        if pool:
            pool.shutdown()
    full_step_ms = 1e3 * statistics.mean(secs)
    value = _step_osc_steps(_step_units()) / (full_step_ms / 1e3)
    batched_osc = sum(sp["n"] for sp in W.batched_systems(BATCH_SYSTEMS, seed=1234))
    return {
        "impl": "reference",
        "metric": "oscillator-steps/s (fused LD+RNG, all generators, whole hot path)",
        "value": value, "unit": "oscillator-steps/s", "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": 1e3 * wall / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32+u32",
        "data": "synthetic (seeded oscillators; equilibrium start)",
        "config": bench_config(world, batched_osc),
        "cpu_baseline": {"value": value, "unit": "oscillator-steps/s", "cores": workers,
                         "cpu": host_cpu(), "kind": "oracle",
                         "sample": _sample_text(scale, workers),
                         "full_step_ms_extrapolated": full_step_ms},
        "e2e": {"value": value, "unit": "oscillator-steps/s", "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
    }


CASES = ("ld_taus", "ld_ran2", "ld_lagfib", "fill_uniform_taus", "fill_normal_taus",
         "fill_uniform_ran2", "fill_normal_ran2", "fill_uniform_lagfib", "fill_normal_lagfib",
         "batched_taus", "adjoint_taus", "adjoint_ran2", "ld_taus_1e8", "ld_ran2_1e8",
         "ld_lagfib_1e8")


def run_case(name: str):
    """Short launches of one part (for profiler captures): fused runs use the
    bench's 1e6 oscillators x 100 steps (x and v: 24 MB), fills 2^28 numbers
    (1 GiB, larger than L2)."""
    import torch
    from paper_1003_1123_gb300 import gbrng as G
    kind = part_kind(name)
    if name.startswith("adjoint_"):
        # the bench's adjoint system (1e5 oscillators), 1000 steps, checkpoints
        # every 100, noise regenerated as in the bench step
        r = G.rng_init(kind, SEED + 11, ADJ_N)
        x = torch.zeros((ADJ_N, 3), dtype=torch.float32, device="cuda")
        s = G.LdSystem(r, x, torch.zeros_like(x), K_per=torch.ones(ADJ_N, device="cuda"),
                       **{k: v for k, v in PARAMS.items() if k != "K"})
        G.ld_init_equilibrium(s)
        G.ld_set_adjoint_history_limit(0)
        for _ in range(2):
            G.ld_backward(s, 1000, ADJ_CKPT)
    elif name.endswith("_1e8"):
        # the large workload at 1e7 oscillators (x, v 240 MB, larger than L2) x 10 steps
        n = 10**7
        r = G.rng_init(kind, SEED, n)
        x = torch.zeros((n, 3), dtype=torch.float32, device="cuda")
        s = G.LdSystem(r, x, torch.zeros_like(x), **LARGE_PARAMS)
        G.ld_init_equilibrium(s)
        for _ in range(2):
            G.ld_run(s, 10)
    elif name == "batched_taus":
        # the bench's 512 systems; the second graph replay (autotuned shape
        # cached by the first) runs inside the NVTX range "profile"
        systems = []
        for sp in W.batched_systems(BATCH_SYSTEMS, seed=1234):
            r = G.rng_init("taus", sp["seed"], sp["n"])
            x = torch.zeros((sp["n"], 3), dtype=torch.float32, device="cuda")
            s = G.LdSystem(r, x, torch.zeros_like(x), K=sp["K"], m=sp["m"], gamma=sp["gamma"],
                           kT=sp["kT"], dt=sp["dt"])
            G.ld_init_equilibrium(s)
            systems.append(s)
        G.ld_run_batched(systems, BATCH_STEPS)
        torch.cuda.synchronize()
        torch.cuda.nvtx.range_push("profile")
        G.ld_run_batched(systems, BATCH_STEPS)
        torch.cuda.synchronize()
        torch.cuda.nvtx.range_pop()
    elif name.startswith("ld_"):
        n = N_OSC
        r = G.rng_init(kind, SEED, n)
        x = torch.zeros((n, 3), dtype=torch.float32, device="cuda")
        v = torch.zeros_like(x)
        s = G.LdSystem(r, x, v, **PARAMS)
        G.ld_init_equilibrium(s)
        for _ in range(2):
            G.ld_run(s, 100)
    else:
        r = G.rng_init(kind, SEED, N_OSC)
        out = torch.empty(2**28, dtype=torch.float32, device="cuda")
        f = G.rng_fill_uniform if "uniform" in name else G.rng_fill_normal
        for _ in range(2):
            f(r, 2**28, out=out)
    torch.cuda.synchronize()
    print(f"case {name} done")


def run_sweep():
    """Time per 1000 steps against N for every generator (Hybrid Taus, Ran2,
    Lagged Fibonacci and the LCG), persistent and paper form (one launch per
    step), the state bytes per generator, and the share of
    a fused step that generating its numbers alone takes (a fill of the same
    count of normals).  Prints one JSON object; not the bench line."""
    import torch
    from paper_1003_1123_gb300 import gbrng as G
    steps = 1000
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]

    def timed(fn):
        fn()
        torch.cuda.synchronize()
        ev[0].record()
        fn()
        ev[1].record()
        torch.cuda.synchronize()
        return ev[0].elapsed_time(ev[1])

    clocks = Clocks(torch.cuda.current_device())
    clocks.start()
    rows = []
    for n in (10**3, 10**4, 10**5, 10**6, 10**7, 10**8):
        for kind in KINDS + ("lcg",):
            r = G.rng_init(kind, SEED, n)
            x = torch.zeros((n, 3), dtype=torch.float32, device="cuda")
            v = torch.zeros_like(x)
            s = G.LdSystem(r, x, v, **PARAMS)
            G.ld_init_equilibrium(s)
            row = {"n": n, "kind": kind, "state_bytes": G.rng_state_bytes(r),
                   "xv_bytes": 24 * n,
                   "persistent_ms_per_1000": timed(lambda: G.ld_run(s, steps, stats=False))}
            if n > 10**7:
                row["paper_form_ms_per_1000"] = None    # minutes at this size; see 1e7
            else:
                try:
                    row["paper_form_ms_per_1000"] = timed(
                        lambda: G.ld_run_stepwise(s, steps, stats=False))
                except G.GbrngError as e:
                    row["paper_form_ms_per_1000"] = None
                    row["paper_form"] = str(e)[:120]
            # the numbers of fill_steps steps (at most 4e8 floats), scaled to 1000 steps
            fill_steps = max(1, min(steps, 10**8 // n))
            nums = 4 * n * fill_steps
            out = torch.empty(nums, dtype=torch.float32, device="cuda")
            f = G.rng_init(kind, SEED + 1, n)
            row["fill_normal_ms_same_numbers"] = (timed(lambda: G.rng_fill_normal(f, nums, out=out))
                                                  * steps / fill_steps)
            row["rng_share_of_fused"] = (row["fill_normal_ms_same_numbers"]
                                         / row["persistent_ms_per_1000"])
            del out, f
            rows.append(row)
            del s, x, v, r
            torch.cuda.empty_cache()
    # every Table I row at N = 1000 oscillators (row 0: 4N > 2(ll - sl), several rounds a step)
    lag_rows = []
    for row in range(10):
        r = G.rng_init_lfg(SEED, 1000, lag_row=row)
        x = torch.zeros((1000, 3), dtype=torch.float32, device="cuda")
        s = G.LdSystem(r, x, torch.zeros_like(x), **PARAMS)
        G.ld_init_equilibrium(s)
        sl, ll = G.rng_lfg_lags(row)
        # three rounds of the deepest fan (K of 16, 8, 4, 2 with K (ll - sl) <= 4.1e6)
        k = next((k for k in (16, 8, 4) if k * (ll - sl) <= 4100000), 2)
        d = ll - sl
        ring = (max(3 * k * d, (k + 1) * d + k * sl) + 31) // 32 * 32
        lag_rows.append({"row": row, "sl": sl, "ll": ll, "ring_bytes": 4 * ring,
                         "portable_state_bytes": G.rng_state_bytes(r),
                         "ms_per_1000": timed(lambda: G.ld_run(s, steps, stats=False))})
        del s, x, r
    # Lagged Fibonacci systems beyond the SMs' shared memory, even and odd N (their x and v
    # rows change alignment from step to step), one spring constant and one each
    stream_rows = []
    for n in (1200000, 1200001, 10**7, 10**7 + 1):
        for per_k in (False, True):
            r = G.rng_init("lagfib", SEED, n)
            x = torch.zeros((n, 3), dtype=torch.float32, device="cuda")
            K = torch.linspace(0.5, 2.0, n, device="cuda") if per_k else None
            s = G.LdSystem(r, x, torch.zeros_like(x), K_per=K, **PARAMS)
            G.ld_init_equilibrium(s)
            stream_rows.append({"n": n, "K_per": per_k,
                                "ms_per_1000": timed(lambda: G.ld_run(s, steps, stats=False))})
            del s, x, r, K
    torch.cuda.empty_cache()
    # the overdamped 1-D test of Sec. IV (Eq. 4-5) at the paper's parameters
    # (k_sp = 0.01 pN/nm, T = 300 K, D = 0.25 nm^2/ns, dt = 1 ps, R0 = 10 nm):
    # 1000 steps with a record every 100, at the paper's N = 1e4 and at 1e6
    kT_ou = 1.380649e-2 * 300.0   # pN nm
    ou_params = dict(k_sp=0.01, xi=kT_ou / 0.25, kT=kT_ou, dt=1e-3)
    ou = []
    for n in (10**4, 10**6):
        for kind in KINDS + ("lcg",):
            r = G.rng_init(kind, SEED + 2, n)
            R = torch.full((n,), 10.0, dtype=torch.float32, device="cuda")
            o = G.OuSystem(r, R, **ou_params)
            ms = timed(lambda: G.ou_run(o, steps, every=100))
            ou.append({"n": n, "kind": kind, "ms_per_1000": ms,
                       "particle_steps_per_s": n * steps / (ms * 1e-3)})
            del o, R, r
    return {"sweep": "time per 1000 steps vs N (E2), state bytes (E3), RNG share (E4), "
                     "Table I rows at N = 1000, streamed Lagged Fibonacci runs, overdamped runs (Sec. IV)",
            "params": PARAMS, "rows": rows, "lag_rows": lag_rows,
            "stream_rows": stream_rows, "ou_params": ou_params,
            "ou": ou, "clocks": clocks.stop()}


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="gbrng", choices=["gbrng", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--case", choices=CASES, help="run one small launch of one part and exit")
    ap.add_argument("--sweep", action="store_true",
                    help="print the N sweep (time per 1000 steps, state bytes) and exit")
    args = ap.parse_args()
    if args.case:
        run_case(args.case)
        return
    if args.sweep:
        print(json.dumps(run_sweep()))
        return
    if args.warmup < 3:
        ap.error("--warmup must be >= 3")

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    dist = None
    if args.impl == "reference":
        if rank != 0:
            return
        print(json.dumps(run_reference(args, world)))
        return
    if world > 1:
        import torch
        import torch.distributed as dist
        torch.cuda.set_device(int(os.environ.get("LOCAL_RANK", 0)))
        dist.init_process_group("nccl")
    line = run_gpu(args, rank, world, dist)
    if rank == 0:
        print(json.dumps(line))
    if dist:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
