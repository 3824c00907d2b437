"""Throughput of batched fire-spread simulations on GB300.

Default step (the largest single-GPU configuration): the uneven batch of
nine synthetic fires on grids from 200 x 300 to 2000 x 1500 cells (10.9 M
cells in total), 100,000 simulations with parameters drawn from the
Uniform[-30, 30] initial distribution of Table 1, all in one persistent
launch replayed as a CUDA graph, each run to extinction and scored against
its fire's reference burnt map (Eq. 2 counts fused in the simulation
kernel, fitness ratios by a second kernel).  Inputs are resident on the
device before timing; every step uses fresh seeds; L2 is flushed (256 MB
write) before every timed step.

``--workload ga512``: one GA generation of the 512 x 512 calibration
workload (256 Gauss(0, 5) parameter vectors x 16 replicates).
``--workload recover``: parameter recovery of the plain GA (populations 256
and 1024) and the surrogate-screened GA against the reference parameters.
``--impl reference``: the CPU oracle on the same workload and sample as the
``cpu_baseline`` leg of the default line.

Prints one JSON line.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

from paper_1701_03549_gb300 import parallel, synth, workloads  # noqa: E402

METRIC = "CA sims/s"
UNIT = "sims/s"
POP, REPS = 256, 16
SIMS = POP * REPS
# Algorithmic operations of one trial (one decision of a burning neighbour
# against its target): a quarter of a Philox4x32-10 block, about 25 integer
# operations per 32-bit word (10 rounds of two 32x32->64 multiplies, the
# xors and the key schedule, over four words), plus about 15 single-precision
# operations for Eq. 1 in one direction, the logistic and the comparison
# with the draw.
OPS_PER_TRIAL = 40
ALU_LANES_PER_SM = 128
UNEVEN = ("uneven_fires: nine fires on 200x300 ... 2000x1500 grids (10.9 M "
          "cells), 100,000 simulations in one persistent launch (11,112 on "
          "the first fire, 11,111 on each other), Uniform[-30,30] parameters, "
          "centre ignitions, targets from the reference parameters")
GA512 = ("ga_generation_512: 512x512 map, 256 Gauss(0,5) parameter "
         "vectors x 16 replicates = 4096 simulations/step, centre "
         "ignition, constant 45 deg wind, target from the reference "
         "parameters")
L2_NOTE = "flushed before every timed step (256 MB write)"
# Stratified oracle samples (the same in cpu_baseline and --impl reference)
UNEVEN_PER_FIRE = 16


def _peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(p) as f:
            return json.load(f), "measured"
    except OSError:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0,
                "sm_max_mhz": 2070.0}, "fallback"


def _strip_comments(src: str) -> str:
    """C/C++ source without its comments and blank-line runs (string and
    character literals kept), so that a record of the kernel's counters stays
    valid across edits of its comments only."""
    import re

    pat = re.compile(r'//[^\n]*|/\*.*?\*/|"(?:\\.|[^"\\])*"|\'(?:\\.|[^\'\\])*\'',
                     re.S)
    out = pat.sub(lambda m: m.group(0) if m.group(0)[0] in "\"'" else " ", src)
    lines = [ln.rstrip() for ln in out.splitlines()]
    return "\n".join(ln for ln in lines if ln.strip())


def _kernel_hash():
    """SHA-256 of the simulation kernel's sources (code only, comments
    stripped): the key of the committed ncu records."""
    h = hashlib.sha256()
    for f in ("fire_kernels.cu", "fire_device.cuh", "fire_internal.h"):
        with open(os.path.join(ROOT, "paper_1701_03549_gb300", "csrc", f),
                  encoding="utf-8") as fh:
            h.update(_strip_comments(fh.read()).encode())
    return h.hexdigest()


def _committed_profile(name="k_simulate_traffic.json"):
    """The committed ncu record of the simulation kernel (DRAM and L2 bytes
    per launch), or None when the kernel changed since it was captured."""
    p = os.path.join(ROOT, "profiles", name)
    try:
        with open(p) as f:
            d = json.load(f)
    except OSError:
        return None
    if d.get("source_sha256") != _kernel_hash():
        return None
    return d


def _committed_traffic():
    d = _committed_profile()
    return None if d is None else d.get("dram_bytes_per_launch")


def _memory_roofs(kernel_s, peaks, peaks_kind, name="k_simulate_traffic.json"):
    """DRAM and L2 bandwidth of the simulation kernel: bytes per launch from
    the committed ncu capture over the event-timed launch duration, against
    the measured HBM copy bandwidth and ncu's L2 sector peak."""
    d = _committed_profile(name)
    if d is None:
        return None
    dram = d["dram_bytes_per_launch"] / kernel_s / 1e9
    l2 = d["l2_bytes_per_launch"] / kernel_s / 1e9
    l2_peak = (d["l2_bytes_per_launch"] / (d["ncu_duration_ms"] / 1e3) / 1e9 /
               (d["l2_pct_of_peak_sectors"] / 100.0))
    hbm = float(peaks.get("hbm_gbs", 6800.0))
    return {"dram_gbs": dram, "dram_frac": dram / hbm,
            "dram_peak_gbs": hbm, "dram_peak_source": f"hbm_gbs ({peaks_kind})",
            "l2_gbs": l2, "l2_frac": l2 / l2_peak, "l2_peak_gbs": l2_peak,
            "l2_peak_source": "ncu lts__t_sectors peak"}


def _dense_sweep_roof(cell_updates_per_s, peaks, peaks_kind):
    """Cell-updates/s (dense-equivalent: steps x H x W per second) against
    what a dense sweep of the whole grid every step could reach at the
    measured HBM bandwidth, streaming only the 2-bit state (2 bits read and 2
    written per cell-update, 0.5 B) and nothing else.  A reference point for
    the rate, not this kernel's bound: the worklists skip quiet tiles, so
    the kernel moves far fewer bytes than such a sweep."""
    hbm = float(peaks.get("hbm_gbs", 6800.0))
    dense = hbm * 1e9 / 0.5
    return {"model": "dense 2-bit-state sweep, 0.5 B per cell-update",
            "dense_rate": dense, "unit": "cell-updates/s",
            "ratio": cell_updates_per_s / dense,
            "dense_rate_source": f"hbm_gbs ({peaks_kind})"}


class Clocks:
    """nvidia-smi sampling during the timed region."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,"
              "clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.proc = None
        self.path = None
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(index),
                 f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "200"], stdout=open(self.path, "w"),
                stderr=subprocess.DEVNULL)
        except (OSError, FileNotFoundError):
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        with open(self.path) as f:
            lines = f.readlines()
        os.unlink(self.path)
        return self.summarise(lines)

    @staticmethod
    def summarise(lines):
        """Median and maximum SM clock and the throttle reasons seen, from
        the sampler's CSV rows (malformed rows are skipped)."""
        rows = []
        for line in lines:
            parts = [x.strip() for x in line.split(",")]
            if len(parts) != 7:
                continue
            try:
                rows.append((float(parts[0]), float(parts[1]), parts[3:]))
            except ValueError:
                continue
        if not rows:
            return None
        names = ("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown",
                 "sw_power_cap")
        reasons = sorted({names[i] for _, _, r in rows for i, v in enumerate(r)
                          if v.lower() in ("active", "1", "yes")})
        return {"sm_mhz": statistics.median(r[0] for r in rows),
                "sm_max_mhz": max(r[1] for r in rows),
                "reasons": reasons, "samples": len(rows)}


# ---------------------------------------------------------------------------
# The CPU oracle legs: cpu_baseline of the native line and --impl reference.
# Both time the same stratified sample of the workload with the oracle as it
# stands (single-threaded, one simulation per task) on every host core, with
# the targets simulated by the oracle itself, and extrapolate per fire.

_WORKER = {}


def _lands(kind):
    if kind == "uneven":
        return workloads.uneven_lands()
    return [synth.preset_landscape("ga_generation_512")]


def _oracle_init(kind, packed, barrier):
    """Spawned worker: the oracle's covariates of every map of the workload
    and, for timing jobs, the targets (bit-packed)."""
    import oracle

    lands = _lands(kind)
    _WORKER["F"] = [oracle.Features(L) for L in lands]
    _WORKER["ign"] = [synth.centre_ignition(L.veg) for L in lands]
    _WORKER["burnable"] = [int((L.veg != 0).sum()) for L in lands]
    _WORKER["T"] = (None if packed is None else
                    [np.unpackbits(p, count=L.veg.size).reshape(L.veg.shape)
                     .astype(bool) for p, L in zip(packed, lands)])
    _WORKER["barrier"] = barrier


def _oracle_ready(_):
    """Returns once every worker of the pool has been initialised."""
    _WORKER["barrier"].wait(timeout=600)
    return 0


def _oracle_target_job(j):
    """The reference fire of map j (reference parameters, the first target
    seed whose fire burns enough), simulated by the oracle."""
    F, ign = _WORKER["F"][j], _WORKER["ign"][j]
    seed, burnt = workloads.pick_target(
        lambda s: F.simulate(synth.TRUTH_BETA, ign, s)[1] >= 0,
        _WORKER["burnable"][j])
    return seed, np.packbits(burnt.ravel())


def _oracle_job(args):
    """One oracle simulation: (map index, single-core seconds, steps)."""
    j, beta, ign, seed = args
    t0 = time.perf_counter()
    res, _ = _WORKER["F"][j].simulate(beta, ign, int(seed),
                                      target=_WORKER["T"][j], want_steps=False)
    return j, time.perf_counter() - t0, res["steps"]


class OracleLeg:
    """A spawn pool of single-threaded oracle workers, one per host core,
    holding every map of the workload and the targets the oracle simulated
    for them."""

    def __init__(self, kind: str, cores: int):
        import multiprocessing as mp

        self.kind, self.cores = kind, cores
        nmaps = len(_lands(kind))
        mpc = mp.get_context("spawn")
        with mpc.Pool(min(cores, nmaps), initializer=_oracle_init,
                      initargs=(kind, None, None)) as pool:
            got = pool.map(_oracle_target_job, range(nmaps), chunksize=1)
        self.target_seeds = [int(g[0]) for g in got]
        barrier = mpc.Barrier(cores)
        self.pool = mpc.Pool(cores, initializer=_oracle_init,
                             initargs=(kind, [g[1] for g in got], barrier))
        self.pool.map(_oracle_ready, range(cores), chunksize=1)

    def run(self, jobs):
        t0 = time.perf_counter()
        out = self.pool.map(_oracle_job, jobs, chunksize=1)
        return out, time.perf_counter() - t0

    def close(self):
        self.pool.close()
        self.pool.join()


def _oracle_workload(kind):
    """(workload, sample indices, simulations per map in one step, sample
    description) of the oracle legs: seeds of the first generation/step."""
    if kind == "uneven":
        wl = workloads.uneven_fires()
        idx = workloads.stratified_sample(wl.map_of_sim, UNEVEN_PER_FIRE)
        counts = np.bincount(wl.map_of_sim, minlength=len(wl.lands))
        desc = (f"{UNEVEN_PER_FIRE} simulations per fire ({idx.size}), evenly "
                "spaced over each fire's block of the 100,000-simulation "
                "batch, seeds of the first step; extrapolated per fire: "
                "batch time = sum over fires of (simulations of the fire x "
                "mean single-core seconds of its sampled simulations) / cores")
        mos = wl.map_of_sim
    else:
        wl = workloads.ga_generation_512(POP, REPS)
        idx = np.arange(0, SIMS, REPS, dtype=np.int64)
        counts = np.array([SIMS])
        desc = ("replicate 0 of each of the 256 parameter vectors of the "
                "first generation (256 simulations); extrapolated: "
                "generation time = 4096 x mean single-core seconds / cores")
        mos = np.zeros(wl.n, np.int32)
    jobs = [(int(mos[i]), wl.params[i], tuple(int(v) for v in wl.ignitions[i]),
             int(wl.seeds[i])) for i in idx]
    return wl, jobs, counts, desc


def _extrapolate(results, counts, cores):
    """Seconds of one whole step on `cores` workers: per map, the mean
    single-core seconds of its sampled simulations times its simulations in
    the step, summed, over the cores (perfectly balanced work)."""
    by = {}
    for j, sec, _ in results:
        by.setdefault(j, []).append(sec)
    return sum(counts[j] * float(np.mean(v)) for j, v in by.items()) / cores


def cpu_baseline(kind, cores):
    """The native line's cpu_baseline: the stratified sample once."""
    leg = OracleLeg(kind, cores)
    try:
        wl, jobs, counts, desc = _oracle_workload(kind)
        res, wall = leg.run(jobs)
    finally:
        leg.close()
    est = _extrapolate(res, counts, cores)
    return {"value": int(counts.sum()) / est, "unit": UNIT, "cores": cores,
            "kind": "oracle", "sample": desc,
            "sample_wall_s": round(wall, 2),
            "target_seeds": leg.target_seeds}


def _config(kind, world):
    """The workload as both arms name it (no launch details: those are the
    native arm's own, under "launch")."""
    if kind == "uneven":
        cells = int(sum(H * W for H, W in synth.uneven_fire_shapes()))
        return {"workload": UNEVEN, "sims_per_step": 100_000,
                "cells_total": cells, "graph": True, "l2": L2_NOTE,
                "parallelism": f"replicas x{world}"}
    return {"workload": GA512, "H": 512, "W": 512, "sims_per_step": SIMS,
            "l2": L2_NOTE, "order": "longest-first by predicted spread "
            "(FIRE_LONGEST_FIRST)", "parallelism": f"replicas x{world}"}


def run_reference(args):
    """The oracle arm: W untimed warm-up rounds, then K timed steps that
    cycle through the stratified sample (every sampled simulation at least
    once when K divides it; the value extrapolates from all of them)."""
    rank, world, _ = parallel.env_rank()
    if rank != 0:
        return 0
    kind = "ga512" if args.workload == "ga512" else "uneven"
    cores = os.cpu_count() or 1
    leg = OracleLeg(kind, cores)
    try:
        wl, jobs, counts, desc = _oracle_workload(kind)
        trivial = (0, np.full(5, -1000.0), jobs[0][2], 1)
        for _ in range(args.warmup):
            leg.run([trivial] * cores)
        per = -(-len(jobs) // args.steps)
        timed, walls = [], []
        for k in range(args.steps):
            step = [jobs[(k * per + i) % len(jobs)] for i in range(per)]
            res, wall = leg.run(step)
            timed += res
            walls.append(wall)
    finally:
        leg.close()
    est = _extrapolate(timed, counts, cores)
    value = int(counts.sum()) / est
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT,
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": 1e3 * est, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "u32",
        "data": "synthetic", "config": _config(kind, world),
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores,
                         "kind": "oracle",
                         "sample": desc + f"; the {len(jobs)} sampled "
                                   f"simulations cycled over the {args.steps}"
                                   f" timed steps ({per} per step)",
                         "sample_wall_s": round(sum(walls), 2),
                         "target_seeds": leg.target_seeds},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line))
    return 0


# ---------------------------------------------------------------------------
# Native arm, shared pieces

def _setup_gpu():
    import torch

    rank, world, local = parallel.env_rank()
    if world > 1:
        import torch.distributed as dist

        dist.init_process_group("nccl" if torch.cuda.is_available() else "gloo")
    if not torch.cuda.is_available():
        return None
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    import __graft_entry__

    __graft_entry__.build()
    from paper_1701_03549_gb300 import fire

    stream = torch.cuda.Stream(dev)
    torch.cuda.set_stream(stream)
    ctx = fire.Context(local, stream)
    return torch, fire, ctx, dev, stream, rank, world, local


def _gpu_target(fire, m, ign, burnable):
    """The map's reference fire simulated on this GPU (the first target seed
    whose fire burns enough)."""
    def sim(seed):
        _, bs = m.simulate_batch(np.asarray([synth.TRUTH_BETA]),
                                 np.asarray([ign], np.int32),
                                 np.asarray([seed], np.uint64),
                                 want_steps=True)
        return bs[0] >= 0

    return workloads.pick_target(sim, burnable)


def _alu_roof(torch, dev, trials_per_launch, launch_s):
    peaks, kind = _peaks()
    sm_max = float(peaks.get("sm_max_mhz", 2070.0))
    props = torch.cuda.get_device_properties(dev)
    peak = props.multi_processor_count * ALU_LANES_PER_SM * sm_max * 1e6
    achieved = trials_per_launch * OPS_PER_TRIAL / launch_s
    return peaks, kind, {
        "bound": "alu", "achieved": achieved / 1e12, "peak": peak / 1e12,
        "unit": "Tops/s", "frac": achieved / peak, "kernel": "k_simulate",
        "peak_source": f"{props.multi_processor_count} SMs x "
                       f"{ALU_LANES_PER_SM} lanes x {sm_max:.0f} MHz "
                       f"({kind} max SM clock)",
        "ops_per_trial": OPS_PER_TRIAL, "trials_per_launch": trials_per_launch,
        "kernel_ms": 1e3 * launch_s}


def _pinned(torch, a):
    return torch.from_numpy(np.ascontiguousarray(a)).pin_memory().numpy()


# ---------------------------------------------------------------------------
# Native arm, default step: the nine-fire uneven batch

def _forced_launch(args, ctx):
    """The launch shape given by --launch W,B,Q,S (warps per block, blocks
    per SM, queue entries, state mode), set on the context in place of the
    autotuner's pick (profiling a reduced batch in the shape the full batch
    runs in); None without the option."""
    if not args.launch:
        return None
    w, b, q, st = (int(v) for v in args.launch.split(","))
    ctx.set_launch(w, b, q, st)
    return {"warps_per_block": w, "blocks_per_sm": b, "queue_entries": q,
            "state_mode": st, "ms": None, "forced": True}


def run_uneven(args):
    """One fire_simulate_multi call per step (CUDA-graph replay of the
    ordering kernels and the persistent simulation launch) plus the fitness
    kernel, all on device-resident inputs."""
    g = _setup_gpu()
    if g is None:
        print(json.dumps({"metric": METRIC, "error": "no CUDA device"}))
        return 1
    torch, fire, ctx, dev, stream, rank, world, local = g
    nsteps = args.warmup + args.steps
    n = 100_000
    wl = workloads.uneven_fires(n, first_seed=1 + rank * n * (nsteps + 1))
    if args.sample > 1:   # a reduced batch (profiling): every K-th simulation
        keep = np.arange(0, n, args.sample)
        wl = workloads.MultiWorkload(wl.name, wl.lands, wl.map_of_sim[keep],
                                     wl.params[keep], wl.ignitions[keep],
                                     wl.seeds[keep])
        n = wl.n
    maps = [ctx.landscape_upload(L) for L in wl.lands]
    tseeds = []
    for j, (m, L) in enumerate(zip(maps, wl.lands)):
        ign = tuple(int(v) for v in wl.ignitions[np.argmax(wl.map_of_sim == j)])
        ts, tg = _gpu_target(fire, m, ign, int((L.veg != 0).sum()))
        m.target_upload(tg)
        tseeds.append(int(ts))
    # launch shape: the autotuner times its candidates on a stratified tenth
    # of the batch (outside the timed region) and the library keeps the best
    sub = np.arange(0, n, 10)
    tuned = _forced_launch(args, ctx)
    if tuned is None:
        tuned = fire.fire_autotune(ctx, maps, wl.map_of_sim[sub], wl.params[sub],
                                   wl.ignitions[sub], wl.seeds[sub])
    t_mi = torch.tensor(wl.map_of_sim, device=dev)
    t_p = torch.tensor(wl.params, dtype=torch.float64, device=dev)
    t_g = torch.tensor(wl.ignitions, device=dev)
    t_s = torch.empty(n, dtype=torch.int64, device=dev)
    seeds_host = [wl.seeds + np.uint64(k * n) for k in range(nsteps)]
    seeds_all = [torch.tensor(s.view(np.int64), device=dev) for s in seeds_host]
    out = torch.zeros((n, 6), dtype=torch.int32, device=dev)
    fit = torch.zeros(n, dtype=torch.float64, device=dev)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)
    torch.cuda.synchronize()

    def step(k):
        t_s.copy_(seeds_all[k])
        fire.fire_simulate_multi(ctx, maps, t_mi, t_p, t_g, t_s, device=True,
                                 out=out, graph=True)
        fire.fire_fitness(ctx, out, fire.FITNESS_JACCARD, device=True, out=fit)

    for k in range(args.warmup):
        flush.zero_()
        step(k)
    torch.cuda.synchronize()
    if world > 1:
        torch.distributed.barrier()
    torch.cuda.synchronize()
    clocks = Clocks(local)
    sim_ms, step_ms = [], []
    steps_sum = trials_sum = cells = 0
    sizes = np.array([L.veg.size for L in wl.lands], np.int64)[wl.map_of_sim]
    for j in range(args.steps):
        k = args.warmup + j
        flush.zero_()
        t_s.copy_(seeds_all[k])
        e0, e1, e2 = (torch.cuda.Event(enable_timing=True) for _ in range(3))
        e0.record(stream)
        fire.fire_simulate_multi(ctx, maps, t_mi, t_p, t_g, t_s, device=True,
                                 out=out, graph=True)
        e1.record(stream)
        fire.fire_fitness(ctx, out, fire.FITNESS_JACCARD, device=True, out=fit)
        e2.record(stream)
        torch.cuda.synchronize()
        sim_ms.append(e0.elapsed_time(e1))
        step_ms.append(e0.elapsed_time(e2))
        r = fire.results_view(out)
        assert int((r["status"] & (fire.STATUS_BAD_IGNITION |
                                   fire.STATUS_TIMEOUT)).max()) == 0
        st = r["steps"].astype(np.int64)
        steps_sum += int(st.sum())
        cells += int((st * sizes).sum())
        trials_sum += int(r["trials"].astype(np.int64).sum())
    ck = clocks.stop()
    total_s = parallel.max_over_ranks(sum(step_ms) / 1e3, world, dev)
    value = n * args.steps * world / total_s
    cells_all = parallel.sum_over_ranks(cells, world, dev)
    trials_all = parallel.sum_over_ranks(trials_sum, world, dev)

    # end to end through the C ABI with host buffers (pinned): the same seeds
    # and the same L2 flush as the device-timed steps; each call copies the
    # step's inputs in and its results out, the fitness call copies the
    # results in and the fitness out
    pin_mi = _pinned(torch, wl.map_of_sim)
    pin_p = _pinned(torch, wl.params)
    pin_g = _pinned(torch, wl.ignitions)
    pin_s = [_pinned(torch, s) for s in seeds_host]
    fire.fire_simulate_multi(ctx, maps, pin_mi, pin_p, pin_g, pin_s[0])
    e2e_steps = min(args.steps, 5)
    e2e_s = 0.0
    for j in range(e2e_steps):
        k = args.warmup + j
        flush.zero_()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        res = fire.fire_simulate_multi(ctx, maps, pin_mi, pin_p, pin_g, pin_s[k])
        f = fire.fire_fitness(ctx, res, fire.FITNESS_JACCARD)
        e2e_s += time.perf_counter() - t0
        assert f.shape == (n,)
    e2e_s = parallel.max_over_ranks(e2e_s, world, dev)
    e2e_value = n * e2e_steps * world / e2e_s
    dev_same = parallel.max_over_ranks(sum(step_ms[:e2e_steps]) / 1e3, world,
                                       dev)
    h2d = n * (40 + 8 + 8 + 4) + n * 24
    d2h = n * 24 + n * 8

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline and args.sample == 1:
        cpu = cpu_baseline("uneven", os.cpu_count() or 1)
        cpu["targets_match_gpu"] = cpu["target_seeds"] == tseeds

    if rank == 0:
        launch_s = sum(sim_ms) / len(sim_ms) / 1e3
        peaks, pk, roof = _alu_roof(torch, dev, trials_sum / args.steps,
                                    launch_s)
        uprof = _committed_profile("k_simulate_uneven_traffic.json")
        roof["traffic"] = None if uprof is None else uprof["dram_bytes_per_launch"]
        roof["timed"] = ("the graph (three ordering kernels, counter reset, "
                         "k_simulate), CUDA events on the launching stream")
        roof["memory"] = _memory_roofs(launch_s, peaks, pk,
                                       "k_simulate_uneven_traffic.json")
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": total_s * 1e3 / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "u32", "data": "synthetic",
            "config": dict(_config("uneven", world), **(
                {"sample_every": args.sample, "sims_per_step": n}
                if args.sample > 1 else {})),
            "launch": {k: tuned[k] for k in ("warps_per_block", "blocks_per_sm",
                                             "queue_entries", "state_mode",
                                             "forced") if k in tuned},
            "target_seeds": tseeds,
            "cell_updates_per_s": cells_all / total_s,
            "cell_updates_vs_dense_sweep": _dense_sweep_roof(
                cells_all / total_s, peaks, pk),
            "trials_per_s": trials_all / total_s,
            "mean_steps_per_sim": steps_sum / (n * args.steps),
            "roofline": roof,
            "cpu_baseline": cpu,
            "e2e": {"value": e2e_value, "unit": UNIT,
                    "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h,
                    "steps": e2e_steps,
                    "device_value_same_steps": n * e2e_steps * world / dev_same,
                    "timed": "fire_simulate_multi and fire_fitness on pinned "
                             "host buffers, wall clock per call, with the "
                             "seeds and L2 flush of the first device-timed "
                             "steps"},
            # per step: k_order_count, k_order_scan, k_order_scatter,
            # k_simulate (graph) and k_fitness
            "gpu_launches": 5 * args.steps,
            "clocks": ck,
        }
        print(json.dumps(line))
    for m in maps:
        m.free()
    ctx.close()
    if world > 1:
        torch.distributed.destroy_process_group()
    return 0


# ---------------------------------------------------------------------------
# Native arm, --workload ga512: one GA generation of the 512 x 512 map

def run_ga512(args):
    """fire_simulate_batch in longest-first order plus the fitness kernel on
    device-resident inputs, at the autotuned launch shape."""
    g = _setup_gpu()
    if g is None:
        print(json.dumps({"metric": METRIC, "error": "no CUDA device"}))
        return 1
    torch, fire, ctx, dev, stream, rank, world, local = g
    nsteps = args.warmup + args.steps
    first = parallel.rank_seed_offset(rank, SIMS * (nsteps + 2))
    wl = workloads.ga_generation_512(POP, REPS, first_seed=first)
    if args.sample > 1:   # a reduced batch (profiling): every K-th simulation
        keep = np.arange(0, SIMS, args.sample)
        wl = workloads.Workload(wl.name, wl.land, wl.ignition, wl.params[keep],
                                wl.ignitions[keep], wl.seeds[keep])
    nsim = wl.n
    m = ctx.landscape_upload(wl.land)
    H, W = wl.shape
    tseed, target = _gpu_target(fire, m, wl.ignition,
                                int((wl.land.veg != 0).sum()))
    m.target_upload(target)
    # the autotuner times its candidate shapes on this batch in the step's
    # longest-first order (outside the timed region); the library keeps the
    # fastest
    tuned = _forced_launch(args, ctx)
    if tuned is None:
        tuned = fire.fire_autotune(ctx, [m], None, wl.params, wl.ignitions,
                                   wl.seeds, longest_first=True)
    p_dev = torch.tensor(wl.params, dtype=torch.float64, device=dev)
    g_dev = torch.tensor(wl.ignitions, dtype=torch.int32, device=dev)
    seeds_host = [wl.seeds + np.uint64(k * nsim) for k in range(nsteps)]
    s_dev = [torch.tensor(s.view(np.int64), device=dev) for s in seeds_host]
    outs = [torch.zeros((nsim, 6), dtype=torch.int32, device=dev)
            for _ in range(nsteps)]
    fit = [torch.zeros(nsim, dtype=torch.float64, device=dev)
           for _ in range(nsteps)]
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)
    torch.cuda.synchronize()

    def step(k):
        m.simulate_batch(p_dev, g_dev, s_dev[k], device=True, out=outs[k],
                         longest_first=True)
        fire.fire_fitness(ctx, outs[k], fire.FITNESS_JACCARD, device=True,
                          out=fit[k])

    for k in range(args.warmup):
        flush.zero_()
        step(k)
    torch.cuda.synchronize()
    if world > 1:
        torch.distributed.barrier()
    torch.cuda.synchronize()
    ev = [tuple(torch.cuda.Event(enable_timing=True) for _ in range(3))
          for _ in range(args.steps)]
    clocks = Clocks(local)
    for j in range(args.steps):
        k = args.warmup + j
        flush.zero_()
        e0, e1, e2 = ev[j]
        e0.record(stream)
        m.simulate_batch(p_dev, g_dev, s_dev[k], device=True, out=outs[k],
                         longest_first=True)
        e1.record(stream)
        fire.fire_fitness(ctx, outs[k], fire.FITNESS_JACCARD, device=True,
                          out=fit[k])
        e2.record(stream)
    torch.cuda.synchronize()
    ck = clocks.stop()
    if world > 1:
        torch.distributed.barrier()
    sim_ms = [ev[j][0].elapsed_time(ev[j][1]) for j in range(args.steps)]
    step_ms = [ev[j][0].elapsed_time(ev[j][2]) for j in range(args.steps)]
    total_s = parallel.max_over_ranks(sum(step_ms) / 1e3, world, dev)
    res = [fire.results_view(outs[args.warmup + j]) for j in range(args.steps)]
    steps_sum = sum(int(r["steps"].astype(np.int64).sum()) for r in res)
    trials_sum = sum(int(r["trials"].astype(np.int64).sum()) for r in res)
    steps_all = parallel.sum_over_ranks(steps_sum, world, dev)
    trials_all = parallel.sum_over_ranks(trials_sum, world, dev)
    assert all(int((r["status"] & (fire.STATUS_BAD_IGNITION
                                    | fire.STATUS_TIMEOUT)).max()) == 0
               for r in res)
    value = nsim * args.steps * world / total_s

    # end to end through the C ABI with host buffers (pinned): the same seeds
    # and L2 flush as the device-timed steps
    pin_p = _pinned(torch, wl.params)
    pin_g = _pinned(torch, wl.ignitions)
    pin_s = [_pinned(torch, s) for s in seeds_host]
    m.simulate_batch(pin_p, pin_g, pin_s[0], longest_first=True)
    e2e_steps = min(args.steps, 10)
    e2e_s = 0.0
    for j in range(e2e_steps):
        k = args.warmup + j
        flush.zero_()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        r, _ = m.simulate_batch(pin_p, pin_g, pin_s[k], longest_first=True)
        f = fire.fire_fitness(ctx, r, fire.FITNESS_JACCARD)
        e2e_s += time.perf_counter() - t0
        assert f.shape == (nsim,)
    e2e_s = parallel.max_over_ranks(e2e_s, world, dev)
    e2e_value = nsim * e2e_steps * world / e2e_s
    dev_same = parallel.max_over_ranks(sum(step_ms[:e2e_steps]) / 1e3, world,
                                       dev)
    h2d = nsim * (40 + 8 + 8) + nsim * 24
    d2h = nsim * 24 + nsim * 8

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline and args.sample == 1:
        cpu = cpu_baseline("ga512", os.cpu_count() or 1)
        cpu["targets_match_gpu"] = cpu["target_seeds"] == [int(tseed)]

    if rank == 0:
        launch_s = sum(sim_ms) / len(sim_ms) / 1e3
        peaks, pk, roof = _alu_roof(torch, dev, trials_sum / args.steps,
                                    launch_s)
        roof["traffic"] = _committed_traffic()
        roof["timed"] = ("k_spread_key, k_rank_desc and k_simulate, CUDA "
                         "events on the launching stream")
        roof["memory"] = _memory_roofs(launch_s, peaks, pk)
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * total_s / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "u32", "data": "synthetic",
            "config": dict(_config("ga512", world), **(
                {"sample_every": args.sample, "sims_per_step": nsim}
                if args.sample > 1 else {})),
            "launch": {k: tuned[k] for k in ("warps_per_block", "blocks_per_sm",
                                             "queue_entries", "state_mode",
                                             "forced") if k in tuned},
            "target_seed": int(tseed), "target_cells": int(target.sum()),
            "cell_updates_per_s": steps_all * H * W / total_s,
            "cell_updates_vs_dense_sweep": _dense_sweep_roof(
                steps_all * H * W / total_s, peaks, pk),
            "trials_per_s": trials_all / total_s,
            "mean_steps_per_sim": steps_all / (nsim * args.steps * world),
            "roofline": roof,
            "cpu_baseline": cpu,
            "e2e": {"value": e2e_value, "unit": UNIT,
                    "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h,
                    "steps": e2e_steps,
                    "device_value_same_steps": nsim * e2e_steps * world / dev_same,
                    "timed": "fire_simulate_batch and fire_fitness on pinned "
                             "host buffers, wall clock per call, with the "
                             "seeds and L2 flush of the first device-timed "
                             "steps"},
            # per step: k_spread_key and k_rank_desc (longest-first order),
            # k_simulate, k_fitness
            "gpu_launches": 4 * args.steps,
            "clocks": ck,
        }
        print(json.dumps(line))
    m.free()
    ctx.close()
    if world > 1:
        torch.distributed.destroy_process_group()
    return 0


IGNITION = ("ignition_search_1024: 1024x1024 map (spatially varying wind), "
            "target from the reference parameters at the centre ignition; "
            "32x32 candidate ignitions over the target's bounding box, "
            "snapped to burnt cells, x 64 replicates = 65,536 simulations, "
            "the reference parameters, Jaccard fitness, cutoff 0.3")
SINGLE128 = ("single_fire_128: 128x128 map, constant 45 deg wind, the "
             "reference parameters, centre ignition, 64 replicates, int32 "
             "burn-step maps")


def run_small(args, kind):
    """The two smaller configurations through their public calls: the
    ignition search (one ignition_search call: lattice, 65,536 simulations,
    fitness map and ignition estimate) and the 128 x 128 replicates (one
    fire_simulate_batch with burn-step maps on device buffers).  The ALU
    roofline takes its trial count from the same simulations run as one
    batch."""
    g = _setup_gpu()
    if g is None:
        print(json.dumps({"metric": METRIC, "error": "no CUDA device"}))
        return 1
    torch, fire, ctx, dev, stream, rank, world, local = g
    preset = "ignition_search_1024" if kind == "ignition" else "single_fire_128"
    land = synth.preset_landscape(preset)
    H, W = land.veg.shape
    m = ctx.landscape_upload(land)
    ign0 = synth.centre_ignition(land.veg)
    tseed, target = _gpu_target(fire, m, ign0, int((land.veg != 0).sum()))
    m.target_upload(target)
    beta = np.asarray(synth.TRUTH_BETA, np.float64)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)
    nsteps = args.warmup + args.steps
    first = parallel.rank_seed_offset(rank, 1 << 24)
    if kind == "ignition":
        p = synth.PRESETS[preset]
        LH = LW = p["lattice"]
        reps = p["replicates"]
        n = LH * LW * reps
        _, cells, _ = fire.ignition_search(ctx, m, beta, LH, LW, reps, first,
                                           kind=fire.FITNESS_JACCARD, cutoff=0.3)
        ign = np.repeat(cells.reshape(-1, 2), reps, axis=0).astype(np.int32)
        params = np.tile(beta, (n, 1))
        seeds = np.arange(first, first + n, dtype=np.uint64)
        tuned = _forced_launch(args, ctx) or fire.fire_autotune(
            ctx, [m], None, params, ign, seeds)

        def call(k):
            fire.ignition_search(ctx, m, beta, LH, LW, reps, first + k * n,
                                 kind=fire.FITNESS_JACCARD, cutoff=0.3)
        h2d, d2h = 40, 8 * (LH * LW) + 8 * (LH * LW) + 32
        e2e_call = call
    else:
        n = synth.PRESETS[preset]["n_sims"]
        ign = np.tile(np.asarray(ign0, np.int32), (n, 1))
        params = np.tile(beta, (n, 1))
        seeds = np.arange(first, first + n, dtype=np.uint64)
        tuned = _forced_launch(args, ctx) or fire.fire_autotune(
            ctx, [m], None, params, ign, seeds)
        p_dev = torch.tensor(params, device=dev)
        g_dev = torch.tensor(ign, device=dev)
        s_dev = torch.empty(n, dtype=torch.int64, device=dev)
        out = torch.zeros((n, 6), dtype=torch.int32, device=dev)
        bsd = torch.zeros((n, H, W), dtype=torch.int32, device=dev)
        s_all = [torch.tensor((seeds + np.uint64(k * n)).view(np.int64),
                              device=dev) for k in range(nsteps)]

        def call(k):
            s_dev.copy_(s_all[k])
            m.simulate_batch(p_dev, g_dev, s_dev, device=True, out=out,
                             want_steps=True, burn_step=bsd)
        h2d, d2h = n * 56, n * 24 + n * H * W * 4
        pin_p = _pinned(torch, params)
        pin_g = _pinned(torch, ign)
        pin_s = [_pinned(torch, seeds + np.uint64(k * n)) for k in range(nsteps)]

        def e2e_call(k):
            # host buffers: inputs copied in, results and burn-step maps out
            m.simulate_batch(pin_p, pin_g, pin_s[k], want_steps=True)
    for k in range(args.warmup):
        flush.zero_()
        call(k)
    torch.cuda.synchronize()
    clocks = Clocks(local)
    ev = [(torch.cuda.Event(enable_timing=True),
           torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    wall = 0.0
    for j in range(args.steps):
        flush.zero_()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        ev[j][0].record(stream)
        call(args.warmup + j)
        ev[j][1].record(stream)
        torch.cuda.synchronize()
        wall += time.perf_counter() - t0
    ck = clocks.stop()
    if kind != "ignition":   # end to end through host buffers, same seeds
        wall = 0.0
        for j in range(args.steps):
            flush.zero_()
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            e2e_call(args.warmup + j)
            wall += time.perf_counter() - t0
    dev_s = sum(a.elapsed_time(b) for a, b in ev) / 1e3
    total_s = parallel.max_over_ranks(dev_s, world, dev)
    wall = parallel.max_over_ranks(wall, world, dev)
    value = n * args.steps * world / total_s
    # the same simulations as one batch: trials and kernel time of the
    # ALU roofline
    t_p = torch.tensor(params, device=dev)
    t_g = torch.tensor(ign, device=dev)
    t_s = torch.tensor(seeds.view(np.int64), device=dev)
    t_o = torch.zeros((n, 6), dtype=torch.int32, device=dev)
    m.simulate_batch(t_p, t_g, t_s, device=True, out=t_o)
    flush.zero_()
    e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    e0.record(stream)
    m.simulate_batch(t_p, t_g, t_s, device=True, out=t_o)
    e1.record(stream)
    torch.cuda.synchronize()
    r = fire.results_view(t_o)
    trials = int(r["trials"].astype(np.int64).sum())
    steps_sum = int(r["steps"].astype(np.int64).sum())
    if rank == 0:
        peaks, pk, roof = _alu_roof(torch, dev, trials, e0.elapsed_time(e1) / 1e3)
        roof["traffic"] = None
        roof["timed"] = ("the simulations of one step as one "
                         "fire_simulate_batch launch, CUDA events")
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * total_s / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "u32", "data": "synthetic",
            "config": {"workload": IGNITION if kind == "ignition" else SINGLE128,
                       "H": H, "W": W, "sims_per_step": n, "l2": L2_NOTE,
                       "parallelism": f"replicas x{world}"},
            "launch": {k: tuned[k] for k in ("warps_per_block", "blocks_per_sm",
                                             "queue_entries", "state_mode",
                                             "forced") if k in tuned},
            "target_seed": int(tseed), "target_cells": int(target.sum()),
            "cell_updates_per_s": steps_sum * H * W * args.steps / total_s,
            "trials_per_s": trials * args.steps / total_s,
            "mean_steps_per_sim": steps_sum / n,
            "roofline": roof,
            "cpu_baseline": None,
            "e2e": {"value": n * args.steps * world / wall, "unit": UNIT,
                    "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h,
                    "timed": ("the whole ignition_search call (host outputs), "
                              "wall clock" if kind == "ignition" else
                              "fire_simulate_batch on pinned host buffers "
                              "(parameters, ignitions and seeds in; results "
                              "and burn-step maps out), wall clock per call, "
                              "with the seeds and L2 flush of the "
                              "device-timed steps")},
            "clocks": ck,
        }
        print(json.dumps(line))
    m.free()
    ctx.close()
    return 0


SURROGATE = ("surrogate_screened_ga_1024: 1024x1024 map (spatially varying "
             "wind), target from the reference parameters at the centre "
             "ignition; BF16 surrogate (S=256, ~1.05M params) trained on "
             "200k automaton runs (6250 Gauss(0,5) draws x 16 replicates on "
             "each of the 512x512 and 1024x1024 maps); plain GA population "
             "1024 x 16 replicates against the screened GA (1024 candidates "
             "per generation, 256 simulated x 16 replicates: the 192 best "
             "predicted and 64 drawn from the rest)")
TRAIN_FLOP_PER_PIXEL = 2.0 * 128 * ((144 + 7 * 1152) * 2 + 7 * 1152)
FWD_FLOP_PER_PIXEL = 2.0 * 128 * (144 + 7 * 1152)


def _recovery(ctx, m, ign, hist, truth, f_star, torch, reps=64, frac=0.1,
              tol=0.05, seed=1 << 33):
    """Per generation: the ensemble (best `frac` of the evaluated population)
    mean, its fitness re-scored with `reps` fresh replicates, and the
    relative error of each parameter.  Recovered = the first generation whose
    ensemble fits the target within `tol` of the reference parameters' own
    fitness f_star; returns (fits, errors, generation, seconds) with the
    seconds of the GA up to and including that generation."""
    from paper_1701_03549_gb300 import calibrate, fire

    ens = []
    for P, F in zip(hist.params, hist.fitness):
        order = np.argsort(F, kind="stable")
        ens.append(P[order[:max(1, int(len(F) * frac))]].mean(axis=0))
    ens = np.asarray(ens)
    G = len(ens)
    fits = calibrate.evaluate(
        ctx, m, torch.tensor(ens, device="cuda"), ign,
        np.arange(seed, seed + G * reps, dtype=np.uint64), reps,
        fire.FITNESS_JACCARD, torch).cpu().numpy()
    errs = np.abs(ens - truth) / np.abs(truth)
    t = np.cumsum(hist.seconds)
    hit = np.nonzero(fits <= (1.0 + tol) * f_star)[0]
    g = int(hit[0]) if hit.size else None
    return fits, errs, g, (float(t[g]) if g is not None else None)


def run_surrogate(args):
    """Config 4: surrogate-screened GA against the plain GA (one GPU)."""
    import torch

    import __graft_entry__

    __graft_entry__.build()
    from paper_1701_03549_gb300 import calibrate, fire, surrogate

    rank, world, local = parallel.env_rank()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    stream = torch.cuda.Stream(dev)
    torch.cuda.set_stream(stream)
    ctx = fire.Context(local, stream)
    truth = np.asarray(synth.TRUTH_BETA, np.float64)
    land = synth.preset_landscape("ignition_search_1024")
    land2 = synth.preset_landscape("ga_generation_512")
    m = ctx.landscape_upload(land)
    m2 = ctx.landscape_upload(land2)
    ign = synth.centre_ignition(land.veg)

    def sim_target(seed):
        _, bs = m.simulate_batch(truth[None], np.asarray([ign], np.int32),
                                 np.asarray([seed], np.uint64), want_steps=True)
        return bs[0] >= 0

    _, tgt = workloads.pick_target(sim_target, int((land.veg != 0).sum()))
    m.target_upload(tgt)
    sur = surrogate.Surrogate(ctx, S=256, max_batch=8, seed=1)

    # training data from the automaton
    t0 = time.perf_counter()
    groups = args.train_groups
    data = [surrogate.make_dataset(ctx, m2, land2, sur, groups, 16, 21),
            surrogate.make_dataset(ctx, m, land, sur, groups, 16, 22)]
    torch.cuda.synchronize()
    t_data = time.perf_counter() - t0
    # training
    t0 = time.perf_counter()
    losses = sur.train(data, steps=args.train_steps, lr=2e-3, lr_final=1e-4,
                       seed=3)
    t_train = time.perf_counter() - t0
    pix_per_step = 8 * 256 * 256
    train_tflops = (args.train_steps * pix_per_step * TRAIN_FLOP_PER_PIXEL /
                    t_train / 1e12)
    # forward pass alone (roofline of the convolution path)
    x = torch.empty((8, 256, 256, 16), dtype=torch.bfloat16, device=dev)
    sur.inputs(data[1].planes, 1024, 1024, data[1].params[:8].contiguous(),
               data[1].ign[:8].contiguous(), out=x)
    prob = torch.empty((8, 256, 256), dtype=torch.float32, device=dev)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)
    for _ in range(3):
        sur.net.forward(x, prob)
    ms = []
    for _ in range(10):
        flush.zero_()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        sur.net.forward(x, prob)
        e1.record(stream)
        e1.synchronize()
        ms.append(e0.elapsed_time(e1))
    fwd_ms = statistics.median(ms)
    fwd_tflops = pix_per_step * FWD_FLOP_PER_PIXEL / (fwd_ms / 1e3) / 1e12

    # the two GAs
    gens = args.generations
    clocks = Clocks(local)
    t0 = time.perf_counter()
    plain = calibrate.run_ga(ctx, m, ign, pop=1024, reps=16, generations=gens,
                             ga_seed=5, sim_seed=1 << 30)
    t_plain = time.perf_counter() - t0
    plain256 = calibrate.run_ga(ctx, m, ign, pop=256, reps=16,
                                generations=gens, ga_seed=5,
                                sim_seed=1 << 32)
    t0 = time.perf_counter()
    scr = surrogate.run_screened_ga(ctx, m, land, sur, ign, pop=256, pool=1024,
                                    reps=16, generations=gens, ga_seed=5,
                                    sim_seed=1 << 31)
    t_scr = time.perf_counter() - t0
    ck = clocks.stop()
    f_star = float(calibrate.evaluate(
        ctx, m, torch.tensor(truth[None], device=dev), ign,
        np.arange(1 << 34, (1 << 34) + 64, dtype=np.uint64), 64,
        fire.FITNESS_JACCARD, torch).cpu().numpy()[0])
    f_plain, e_plain, g_plain, s_plain = _recovery(ctx, m, ign, plain, truth,
                                                   f_star, torch)
    f_scr, e_scr, g_scr, s_scr = _recovery(ctx, m, ign, scr, truth, f_star,
                                           torch)
    f_p256, e_p256, g_p256, s_p256 = _recovery(ctx, m, ign, plain256, truth,
                                               f_star, torch)
    peaks, kind = _peaks()
    peak = float(peaks.get("bf16_tflops", 1900.0))
    line = {
        "metric": "time-to-recover 5 params, surrogate-GA vs plain GA",
        "value": s_scr, "unit": "s", "n_gpus": world, "steps": gens,
        "warmup": args.warmup, "ms_per_step": 1e3 * t_scr / gens,
        "higher_is_better": False, "scaling": "weak", "vs_baseline": None,
        "dtype": "bf16 (surrogate) / u32 (automaton)", "data": "synthetic",
        "config": {"workload": SURROGATE, "S": 256, "train_groups": 2 * groups,
                   "train_runs": 2 * groups * 16,
                   "train_steps": args.train_steps, "batch": 8,
                   "recovered_when": "the mean of the best 10% of a generation, "
                                     "re-scored with 64 fresh replicates, fits "
                                     "the target within 5% of the reference "
                                     "parameters' own fitness (64 replicates)"},
        "reference_fitness": f_star,
        "plain_ga": {"generations": gens, "seconds": t_plain,
                     "recovered_generation": g_plain, "recovered_s": s_plain,
                     "sims_per_generation": 1024 * 16,
                     "ensemble_fitness_by_gen": [round(float(x), 4)
                                                 for x in f_plain],
                     "final_rel_error": [round(float(x), 3)
                                         for x in e_plain[-1]]},
        "plain_ga_256": {"generations": gens,
                         "seconds": float(sum(plain256.seconds)),
                         "recovered_generation": g_p256,
                         "recovered_s": s_p256,
                         "sims_per_generation": 256 * 16,
                         "ensemble_fitness_by_gen": [round(float(x), 4)
                                                     for x in f_p256],
                         "final_rel_error": [round(float(x), 3)
                                             for x in e_p256[-1]]},
        "screened_ga": {"generations": gens, "seconds": t_scr,
                        "recovered_generation": g_scr, "recovered_s": s_scr,
                        "sims_per_generation": 256 * 16,
                        "ensemble_fitness_by_gen": [round(float(x), 4)
                                                    for x in f_scr],
                        "final_rel_error": [round(float(x), 3)
                                            for x in e_scr[-1]]},
        "training": {"data_s": t_data, "train_s": t_train,
                     "tflops": train_tflops,
                     "loss_first": float(np.mean(losses[:10])),
                     "loss_last": float(np.mean(losses[-50:]))},
        "roofline": {"bound": "tensor", "achieved": fwd_tflops, "peak": peak,
                     "unit": "TFLOP/s", "frac": fwd_tflops / peak,
                     "traffic": None, "kernel": "surrogate forward "
                     "(k_conv_pair x7, head fused + layer-1 k_conv1), batch 8 x 256^2",
                     "peak_source": f"bf16_tflops ({kind})"},
        "cpu_baseline": None, "e2e": None, "gpu_launches": None,
        "clocks": ck,
    }
    if rank == 0:
        print(json.dumps(line))
    sur.net.free()
    m.free()
    m2.free()
    ctx.close()
    return 0


def run_surrogate_step(args):
    """Surrogate network alone: forward passes and training steps (forward,
    backward, Adam) on a batch of 8 inputs of 256 x 256 (random weights and
    inputs; no automaton), with the tensor-core roofline."""
    import torch

    import __graft_entry__

    __graft_entry__.build()
    from paper_1701_03549_gb300 import fire, surrogate

    rank, world, local = parallel.env_rank()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    stream = torch.cuda.Stream(dev)
    torch.cuda.set_stream(stream)
    ctx = fire.Context(local, stream)
    B, S = 8, 256
    net = fire.Net(ctx, S, B)
    net.set_params(surrogate.init_params(1))
    g = torch.Generator(device=dev).manual_seed(0)
    x = torch.rand((B, S, S, 16), device=dev, generator=g).to(torch.bfloat16)
    t = torch.rand((B, S, S), device=dev, generator=g)
    prob = torch.empty((B, S, S), device=dev)
    loss = torch.zeros(1, dtype=torch.float64, device=dev)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)
    pix = B * S * S

    def timed(fn):
        for _ in range(args.warmup):
            fn()
        ms = []
        for _ in range(args.steps):
            flush.zero_()
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            fn()
            e1.record(stream)
            e1.synchronize()
            ms.append(e0.elapsed_time(e1))
        return statistics.median(ms)

    clocks = Clocks(local)
    fwd_ms = timed(lambda: net.forward(x, prob))
    train_ms = timed(lambda: (net.backward(x, t, loss), net.adam(1e-4)))
    ck = clocks.stop()
    fwd = pix * FWD_FLOP_PER_PIXEL / (fwd_ms / 1e3) / 1e12
    trn = pix * TRAIN_FLOP_PER_PIXEL / (train_ms / 1e3) / 1e12
    peaks, kind = _peaks()
    peak = float(peaks.get("bf16_tflops", 1900.0))
    if rank == 0:
        print(json.dumps({
            "metric": "surrogate training throughput", "value": trn,
            "unit": "TFLOP/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": train_ms,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "bf16", "data": "synthetic",
            "config": {"workload": "surrogate_step: 1.05M-parameter dilated "
                       "conv net, batch 8 x 256 x 256 x 16, random weights "
                       "and inputs", "l2": "flushed between timed steps "
                       "(256 MB write)"},
            "forward_ms": fwd_ms, "forward_tflops": fwd,
            "roofline": {"bound": "tensor", "achieved": trn, "peak": peak,
                         "unit": "TFLOP/s", "frac": trn / peak,
                         "traffic": None, "kernel": "training step (k_conv_pair "
                         "forward and input gradient, k_wgrad_strip, layer-1 "
                         "k_conv1, head, Adam)",
                         "peak_source": f"bf16_tflops ({kind})"},
            "cpu_baseline": None, "e2e": None,
            # per training step: the forward pass (first layer + seven
            # 128 -> 128 convolutions, the head in the last one's epilogue),
            # loss sum and head gradient, per layer a weight and bias gradient
            # (8) and, above the first, an input gradient (7), and Adam
            "gpu_launches": 26 * args.steps,
            "clocks": ck}))
    net.free()
    ctx.close()
    return 0


CROSSOVER_SIDES = (512, 1024, 2048, 4096)
CROSSOVER_REPS = 16   # automaton runs per simulated candidate in the GAs


def _crossover_side(sides, per_sim_ms, target_ms):
    """Map side at which per-simulation time reaches target_ms: log-log
    interpolation between the measured sides (None outside their range)."""
    for k in range(len(sides) - 1):
        a, b = per_sim_ms[k], per_sim_ms[k + 1]
        if a <= target_ms <= b and b > a:
            f = (np.log(target_ms) - np.log(a)) / (np.log(b) - np.log(a))
            return float(np.exp(np.log(sides[k]) +
                                f * (np.log(sides[k + 1]) - np.log(sides[k]))))
    return None


def run_crossover(args):
    """Where the surrogate's screening becomes cheaper than the automaton runs
    it replaces.  Per map side N (square synthetic landscapes, centre
    ignition): the automaton's time per simulation over a batch of prior
    draws Gauss(0, 5) (the screened GA's generation 0) and over the
    reference parameters, one seed each, at one fixed launch shape (4 warps
    x 8 blocks per SM, global state, longest-first order); and the
    surrogate's time per candidate (inputs and forward pass at S = 256,
    chunks of 64) on the same map.  All CUDA-event timed with the L2 flushed
    before every timed call.  A forward pass replaces R automaton runs of
    one candidate (R = 16 in the GAs here): the crossover side is where R
    runs cost as much as one forward pass."""
    g = _setup_gpu()
    if g is None:
        print(json.dumps({"metric": "surrogate crossover", "error": "no CUDA device"}))
        return 1
    torch, fire, ctx, dev, stream, rank, world, local = g
    from paper_1701_03549_gb300 import surrogate

    S, chunk, ncand = 256, 64, 256
    sur = surrogate.Surrogate(ctx, S=S, max_batch=chunk)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)
    ctx.set_launch(4, 8, 3072, fire.STATE_GLOBAL)

    def timed(fn, reps):
        fn()                                   # warm-up (buffers, tables)
        ms = []
        for _ in range(reps):
            flush.zero_()
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            fn()
            e1.record(stream)
            e1.synchronize()
            ms.append(e0.elapsed_time(e1))
        return statistics.median(ms)

    rows = []
    clocks = Clocks(local)
    for N in CROSSOVER_SIDES:
        land = synth.landscape(N, N, seed=31, wind_seed=31)
        m = ctx.landscape_upload(land)
        m.target_upload(np.zeros((N, N), np.uint8))
        ign = np.asarray(synth.centre_ignition(land.veg), np.int32)
        # enough simulations for several per block of the launch
        n = 4096 if N <= 2048 else 2432
        ign_dev = torch.tensor(np.tile(ign, (n, 1)), dtype=torch.int32, device=dev)
        seeds = torch.arange(1, n + 1, dtype=torch.int64, device=dev)
        out = torch.zeros((n, 6), dtype=torch.int32, device=dev)
        row = {"side": N, "simulations": n}
        for name, P in (("prior", surrogate.sample_params(n, 5)),
                        ("reference", np.tile(synth.TRUTH_BETA, (n, 1)))):
            p_dev = torch.tensor(P, dtype=torch.float64, device=dev)

            def sim():
                m.simulate_batch(p_dev, ign_dev, seeds, device=True, out=out,
                                 longest_first=True)

            ms = timed(sim, max(1, args.steps))
            r = fire.results_view(out)
            row[f"automaton_ms_per_sim_{name}"] = ms / n
            row[f"mean_burnt_{name}"] = float(r["burnt"].astype(np.float64).mean())
            row[f"mean_steps_{name}"] = float(r["steps"].astype(np.float64).mean())
        planes = sur.planes(land)
        cp = torch.tensor(surrogate.sample_params(ncand, 6), dtype=torch.float64,
                          device=dev)
        cg = torch.tensor(np.tile(ign, (ncand, 1)), dtype=torch.int32, device=dev)
        ms = timed(lambda: sur.predict(planes, N, N, cp, cg, chunk=chunk),
                   max(1, args.steps))
        row["surrogate_ms_per_candidate"] = ms / ncand
        for name in ("prior", "reference"):
            row[f"forward_in_automaton_runs_{name}"] = (
                row["surrogate_ms_per_candidate"] /
                row[f"automaton_ms_per_sim_{name}"])
        rows.append(row)
        m.free()
        del planes
    ck = clocks.stop()
    ctx.set_launch(0, 0, 0, 0)
    F = statistics.median(r["surrogate_ms_per_candidate"] for r in rows)
    cross = {}
    for name in ("prior", "reference"):
        per = [r[f"automaton_ms_per_sim_{name}"] for r in rows]
        cross[name] = {
            f"R={CROSSOVER_REPS}": _crossover_side(CROSSOVER_SIDES, per,
                                                   F / CROSSOVER_REPS),
            "R=1": _crossover_side(CROSSOVER_SIDES, per, F)}
    if rank == 0:
        print(json.dumps({
            "metric": "map side where one surrogate forward pass costs as much "
                      f"as the {CROSSOVER_REPS} automaton runs it replaces",
            "value": cross["prior"][f"R={CROSSOVER_REPS}"], "unit": "cells",
            "n_gpus": world, "steps": args.steps, "warmup": 1,
            "higher_is_better": False, "scaling": "weak", "vs_baseline": None,
            "dtype": "bf16 (surrogate), f32/f64 screen (automaton)",
            "data": "synthetic",
            "config": {"workload": "crossover: square maps "
                       + ", ".join(f"{N}x{N}" for N in CROSSOVER_SIDES)
                       + "; automaton batches of prior draws and of the "
                       "reference parameters; surrogate S = 256, random "
                       "weights (cost does not depend on them)",
                       "l2": L2_NOTE},
            "crossover_side": cross, "surrogate_ms_per_candidate_median": F,
            "rows": rows, "clocks": ck, "cpu_baseline": None, "e2e": None}))
    sur.net.free()
    ctx.close()
    return 0


BURNOUT = ("burnout_512: the 512x512 GA generation (4096 simulations) with "
           "per-cell burn times: 1 everywhere (the paper's rule) and per fuel "
           "class (1, 3, 1, 2, 4) for classes 0..4, against fire_simulate_batch "
           "at the same launch shape and order")


def run_burnout(args):
    """Burn-time variant of the simulation kernel against the plain one on
    the 512x512 generation (device-resident inputs, L2 flushed before every
    timed call, CUDA events)."""
    g = _setup_gpu()
    if g is None:
        print(json.dumps({"metric": METRIC, "error": "no CUDA device"}))
        return 1
    torch, fire, ctx, dev, stream, rank, world, local = g
    wl = workloads.ga_generation_512(POP, REPS)
    m = ctx.landscape_upload(wl.land)
    tseed, target = _gpu_target(fire, m, wl.ignition,
                                int((wl.land.veg != 0).sum()))
    m.target_upload(target)
    tuned = fire.fire_autotune(ctx, [m], None, wl.params, wl.ignitions,
                               wl.seeds)
    p = torch.tensor(wl.params, dtype=torch.float64, device=dev)
    gi = torch.tensor(wl.ignitions, dtype=torch.int32, device=dev)
    sd = torch.tensor(wl.seeds.view(np.int64), device=dev)
    out = torch.zeros((SIMS, 6), dtype=torch.int32, device=dev)
    ones = torch.ones(wl.land.veg.shape, dtype=torch.uint8, device=dev)
    # the same times with a 2 on one non-burnable cell: the burn-time kernel
    # runs (a batch of ones goes to the plain kernel) with the same fires
    nb = np.argwhere(wl.land.veg == 0)[0]
    ones_k = ones.clone()
    ones_k[int(nb[0]), int(nb[1])] = 2
    fuel = torch.tensor(np.asarray((1, 3, 1, 2, 4), np.uint8)[
        np.minimum(wl.land.veg, 4)], device=dev)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)
    calls = {
        "batch": lambda: m.simulate_batch(p, gi, sd, device=True, out=out),
        "burn_1": lambda: m.simulate_burnout(p, gi, sd, ones, device=True,
                                             out=out),
        "burn_1_in_burn_kernel": lambda: m.simulate_burnout(
            p, gi, sd, ones_k, device=True, out=out),
        "burn_per_fuel": lambda: m.simulate_burnout(p, gi, sd, fuel,
                                                    device=True, out=out),
    }
    res = {}
    clocks = Clocks(local)
    for name, fn in calls.items():
        for _ in range(args.warmup):
            flush.zero_()
            fn()
        ms = []
        for _ in range(args.steps):
            flush.zero_()
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            fn()
            e1.record(stream)
            e1.synchronize()
            ms.append(e0.elapsed_time(e1))
        r = fire.results_view(out)
        res[name] = {"ms": statistics.mean(ms),
                     "mean_steps": float(r["steps"].astype(np.int64).mean()),
                     "trials": int(r["trials"].astype(np.int64).sum())}
    ck = clocks.stop()
    v = SIMS / (res["burn_per_fuel"]["ms"] / 1e3)
    line = {
        "metric": "burn-time CA sims/s", "value": v, "unit": UNIT,
        "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": res["burn_per_fuel"]["ms"], "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "u32",
        "data": "synthetic",
        "config": {"workload": BURNOUT, "l2": L2_NOTE,
                   "launch": {k: tuned[k] for k in (
                       "warps_per_block", "blocks_per_sm", "queue_entries",
                       "state_mode")}},
        "calls": res,
        "burn_1_over_batch": res["burn_1"]["ms"] / res["batch"]["ms"],
        "burn_kernel_1_over_batch": (res["burn_1_in_burn_kernel"]["ms"] /
                                     res["batch"]["ms"]),
        "cpu_baseline": None, "e2e": None,
        "gpu_launches": args.steps * 4, "clocks": ck}
    if rank == 0:
        print(json.dumps(line))
    m.free()
    ctx.close()
    return 0


RECOVER = ("recover_1024: 1024x1024 map (spatially varying wind), target "
           "from the reference parameters (Table 2) at the centre ignition; "
           "plain GA with populations 256 and 1024 x 16 replicates, the "
           "surrogate-screened GA (1024 candidates, 256 simulated x 16) and "
           "the variable-ignition GA (seven genes, population 1024 x 16), 50 "
           "generations each; brute-force Monte Carlo for the time per "
           "simulation")


def _param_errors(hist, truth, frac=0.1):
    """Per generation: the ensemble mean (best `frac` of that generation's
    population) and each parameter's relative error against the truth."""
    ens = []
    for P, F in zip(hist.params, hist.fitness):
        order = np.argsort(F, kind="stable")
        ens.append(P[order[:max(1, int(len(F) * frac))]].mean(axis=0))
    ens = np.asarray(ens)
    k = len(truth)
    return ens, np.abs(ens[:, :k] - truth) / np.abs(truth)


def _time_to_recover(errs, seconds, tol=0.05):
    """GA seconds (cumulative, through the generation) until every
    parameter's relative error is within tol, and per parameter until it
    first is; None where never."""
    t = np.cumsum(seconds)
    allok = np.nonzero((errs <= tol).all(axis=1))[0]
    per = []
    for j in range(errs.shape[1]):
        hit = np.nonzero(errs[:, j] <= tol)[0]
        per.append(None if hit.size == 0 else round(float(t[hit[0]]), 3))
    return (None if allok.size == 0 else round(float(t[allok[0]]), 3)), per


def _ga_report(hist, truth, sims_per_gen):
    ens, errs = _param_errors(hist, truth)
    rec, per = _time_to_recover(errs, hist.seconds)
    return {"seconds": round(float(sum(hist.seconds)), 3),
            "sims_per_generation": sims_per_gen,
            "recovered_all_s": rec, "recovered_each_s": per,
            "rel_error_by_gen": [[round(float(x), 4) for x in e] for e in errs],
            "final_estimate": [round(float(x), 3) for x in ens[-1]],
            "final_rel_error": [round(float(x), 4) for x in errs[-1]]}


RECOVER_MULTI = ("recover_multi_1024: 1024x1024 map (spatially varying "
                 "wind); four reference scars of the reference parameters "
                 "(Table 2) ignited at the burnable cells nearest the quarter "
                 "points, then the points at 1/8, 7/8 and at 3/8, 5/8 of each "
                 "side and the centre (the first four whose fire burns >= 1% "
                 "of the burnable cells for some target seed); "
                 "plain GA population 1024 fitted to the four "
                 "scars at once (4 x 8 replicates per individual) against the "
                 "same GA on the first scar alone (32 replicates), 50 "
                 "generations each, equal automaton runs per generation")


def _nearest_burnable(veg, r, c):
    """Burnable cell nearest (r, c) (Euclidean; ties to the lower index)."""
    cells = np.argwhere(np.asarray(veg) != 0)
    d = (cells[:, 0] - r) ** 2 + (cells[:, 1] - c) ** 2
    return tuple(int(v) for v in cells[int(np.argmin(d))])


def run_recover_multi(args):
    """Parameter recovery from several scars at once (the paper's suggestion
    for parameters a single scar leaves weakly determined, Sec. 4) against
    one scar, at the same number of automaton runs per generation."""
    import torch

    import __graft_entry__

    __graft_entry__.build()
    from paper_1701_03549_gb300 import calibrate, fire

    rank, world, local = parallel.env_rank()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    stream = torch.cuda.Stream(dev)
    torch.cuda.set_stream(stream)
    ctx = fire.Context(local, stream)
    truth = np.asarray(synth.TRUTH_BETA, np.float64)
    land = synth.preset_landscape("ignition_search_1024")
    H, W = land.veg.shape
    # scar ignitions: the burnable cells nearest the quarter points, then the
    # points at 1/8 and 7/8, at 3/8 and 5/8 of each side and the centre,
    # keeping the first four whose reference fire burns at least 1 % of the
    # burnable cells for some target seed (many fires of the reference
    # parameters die out early)
    fr = [(0.25, 0.75), (0.125, 0.875), (0.375, 0.625)]
    pts = [(int(a * H), int(b * W)) for lo, hi in fr
           for a, b in ((lo, lo), (lo, hi), (hi, lo), (hi, hi))]
    pts.append((H // 2, W // 2))
    ignitions, maps, tseeds, sizes = [], [], [], []
    for r, c in pts:
        if len(maps) == 4:
            break
        ign = _nearest_burnable(land.veg, r, c)
        if ign in ignitions:
            continue
        m = ctx.landscape_upload(land)
        try:
            ts, tg = _gpu_target(fire, m, ign, int((land.veg != 0).sum()))
        except RuntimeError:
            m.free()
            continue
        m.target_upload(tg)
        ignitions.append(ign)
        maps.append(m)
        tseeds.append(int(ts))
        sizes.append(int(tg.sum()))
    gens = args.generations
    clocks = Clocks(local)
    multi = calibrate.run_ga_multi(ctx, maps, ignitions, pop=1024, reps=8,
                                   generations=gens, ga_seed=5,
                                   sim_seed=1 << 40)
    single = calibrate.run_ga(ctx, maps[0], ignitions[0], pop=1024, reps=32,
                              generations=gens, ga_seed=5, sim_seed=1 << 41)
    ck = clocks.stop()
    rm = _ga_report(multi, truth, 1024 * 32)
    rs = _ga_report(single, truth, 1024 * 32)
    line = {
        "metric": "time-to-recover 5 params (each within 5% of the reference "
                  "value), plain GA population 1024 fitted to four scars",
        "value": rm["recovered_all_s"], "unit": "s", "n_gpus": world,
        "steps": gens, "warmup": 0,
        "ms_per_step": 1e3 * rm["seconds"] / gens, "higher_is_better": False,
        "scaling": "weak", "vs_baseline": None, "dtype": "u32",
        "data": "synthetic",
        "config": {"workload": RECOVER_MULTI, "ignitions": ignitions,
                   "target_seeds": tseeds, "target_cells": sizes,
                   "reference": list(truth),
                   "estimate": "mean of the best 10% of a generation"},
        "four_scars": rm, "one_scar": rs,
        "cpu_baseline": None, "e2e": None, "gpu_launches": None,
        "clocks": ck,
    }
    if rank == 0:
        print(json.dumps(line))
    for m in maps:
        m.free()
    ctx.close()
    return 0


def run_recover(args):
    """Parameter recovery against the reference parameters (Table 2 layout
    per generation; Table 3 layout for the variable-ignition GA) and the GA
    against Monte Carlo time per simulation (App. C, Fig. 11)."""
    import torch

    import __graft_entry__

    __graft_entry__.build()
    from paper_1701_03549_gb300 import calibrate, fire, surrogate

    rank, world, local = parallel.env_rank()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    stream = torch.cuda.Stream(dev)
    torch.cuda.set_stream(stream)
    ctx = fire.Context(local, stream)
    truth = np.asarray(synth.TRUTH_BETA, np.float64)
    land = synth.preset_landscape("ignition_search_1024")
    land2 = synth.preset_landscape("ga_generation_512")
    m = ctx.landscape_upload(land)
    m2 = ctx.landscape_upload(land2)
    ign = synth.centre_ignition(land.veg)
    tseed, tgt = _gpu_target(fire, m, ign, int((land.veg != 0).sum()))
    m.target_upload(tgt)
    gens = args.generations
    clocks = Clocks(local)
    plain = calibrate.run_ga(ctx, m, ign, pop=1024, reps=16, generations=gens,
                             ga_seed=5, sim_seed=1 << 30)
    plain256 = calibrate.run_ga(ctx, m, ign, pop=256, reps=16,
                                generations=gens, ga_seed=5, sim_seed=1 << 32)
    ga7 = calibrate.run_ga_ignition(ctx, m, tgt, land.veg != 0, pop=1024,
                                    reps=16, generations=gens, ga_seed=5,
                                    sim_seed=1 << 35)
    # brute-force Monte Carlo (App. C): uniform parameters, one replicate
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    n_mc = 1024 * 16
    calibrate.run_mc(ctx, m, ign, n=n_mc, reps=1, seed=11, sim_seed=1 << 36)
    t_mc = time.perf_counter() - t0
    # the surrogate-screened GA (trained on automaton runs of both maps)
    sur = surrogate.Surrogate(ctx, S=256, max_batch=8, seed=1)
    t0 = time.perf_counter()
    data = [surrogate.make_dataset(ctx, m2, land2, sur, args.train_groups, 16,
                                   21),
            surrogate.make_dataset(ctx, m, land, sur, args.train_groups, 16,
                                   22)]
    sur.train(data, steps=args.train_steps, lr=2e-3, lr_final=1e-4, seed=3)
    t_train = time.perf_counter() - t0
    scr = surrogate.run_screened_ga(ctx, m, land, sur, ign, pop=256, pool=1024,
                                    reps=16, generations=gens, ga_seed=5,
                                    sim_seed=1 << 31)
    ck = clocks.stop()
    rp = _ga_report(plain, truth, 1024 * 16)
    r256 = _ga_report(plain256, truth, 256 * 16)
    rscr = _ga_report(scr, truth, 256 * 16)
    rscr["surrogate_training_s"] = round(t_train, 3)
    # variable ignition: Table 3 layout over the best tenth of every
    # individual the GA evaluated
    P7, F7 = ga7.all()
    est = calibrate.ensemble(P7, F7, keep=max(1, len(F7) // 10))
    ref7 = list(truth) + [float(ign[1]), float(ign[0])]
    names = ["b0", "b1", "b2", "b3", "b4", "x", "y"]
    table3 = {nm: {"reference": r, "mean": round(float(mu), 3),
                   "sd": round(float(sd), 3)}
              for nm, r, mu, sd in zip(names, ref7, est["mean"], est["sd"])}
    ens7, err7 = _param_errors(ga7, truth)
    ga_sim_s = sum(plain.seconds) / (gens * 1024 * 16)
    line = {
        "metric": "time-to-recover 5 params (each within 5% of the reference "
                  "value), plain GA population 1024",
        "value": rp["recovered_all_s"], "unit": "s", "n_gpus": world,
        "steps": gens, "warmup": 0,
        "ms_per_step": 1e3 * rp["seconds"] / gens, "higher_is_better": False,
        "scaling": "weak", "vs_baseline": None,
        "dtype": "u32 (automaton) / bf16 (surrogate)", "data": "synthetic",
        "config": {"workload": RECOVER, "target_seed": int(tseed),
                   "reference": list(truth),
                   "estimate": "mean of the best 10% of a generation"},
        "plain_ga_1024": rp, "plain_ga_256": r256, "screened_ga": rscr,
        "variable_ignition_ga": {
            "seconds": round(float(sum(ga7.seconds)), 3),
            "table3": table3, "ensemble_size": est["size"],
            "final_rel_error_beta": [round(float(x), 4) for x in err7[-1]],
            "final_xy": [round(float(x), 2) for x in ens7[-1][5:]],
            "reference_xy": ref7[5:]},
        "ga_vs_mc": {"ga_s_per_sim": ga_sim_s, "mc_s_per_sim": t_mc / n_mc,
                     "ratio": ga_sim_s / (t_mc / n_mc),
                     "note": "wall time per simulation of whole GA "
                             "generations against one Monte Carlo batch of "
                             f"{n_mc} uniform draws (App. C, Fig. 11: the "
                             "paper's GA simulations took about half)"},
        "cpu_baseline": None, "e2e": None, "gpu_launches": None,
        "clocks": ck,
    }
    if rank == 0:
        print(json.dumps(line))
    sur.net.free()
    m.free()
    m2.free()
    ctx.close()
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=("native", "reference"),
                    default="native")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--sample", type=int, default=1,
                    help="time every K-th simulation of the workload only (a "
                         "reduced batch for profiling; not a headline line)")
    ap.add_argument("--workload",
                    choices=("uneven", "ga512", "ignition", "single128",
                             "recover", "recover_multi", "burnout",
                             "surrogate", "surrogate_step", "crossover"),
                    default="uneven",
                    help="uneven (default): nine fires 200x300..2000x1500, "
                         "100k simulations in one launch; ga512: one "
                         "512x512 GA generation; ignition: the 1024x1024 "
                         "ignition search; single128: 64 replicates on "
                         "128x128 with burn-step maps; recover_multi: the "
                         "GA fitted to four scars at once; recover: parameter "
                         "recovery of the GAs; surrogate: the "
                         "surrogate-screened GA against the plain GA; "
                         "surrogate_step: the surrogate network alone; "
                         "crossover: map side where screening pays")
    ap.add_argument("--launch", default="",
                    help="W,B,Q,S: force the simulation launch shape (warps "
                         "per block, blocks per SM, queue entries, state "
                         "mode 1 shared / 2 global) instead of autotuning "
                         "(uneven and ga512; for profiling)")
    ap.add_argument("--generations", type=int, default=50)
    ap.add_argument("--train-steps", type=int, default=1500)
    ap.add_argument("--train-groups", type=int, default=6250)
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        if args.workload not in ("uneven", "ga512"):
            print(json.dumps({"impl": "reference", "unavailable":
                              "the oracle arm times the automaton workloads "
                              "(uneven, ga512) only"}))
            return 0
        return run_reference(args)
    if args.workload == "ga512":
        return run_ga512(args)
    if args.workload in ("ignition", "single128"):
        return run_small(args, args.workload)
    if args.workload == "recover":
        return run_recover(args)
    if args.workload == "recover_multi":
        return run_recover_multi(args)
    if args.workload == "burnout":
        return run_burnout(args)
    if args.workload == "surrogate":
        return run_surrogate(args)
    if args.workload == "surrogate_step":
        return run_surrogate_step(args)
    if args.workload == "crossover":
        return run_crossover(args)
    return run_uneven(args)


if __name__ == "__main__":
    sys.exit(main())
