"""Benchmark: spin-flip attempts/s of augmented PAMC on GB300.

Workload (one GPU): the two sparse Max-Cut instances of the augmented-PAMC
configuration -- a 141x141 toroidal grid (N=19,881, 39,762 edges, +-1 weights)
and a random sparse graph (N=7,000, average degree 5.7, +-1 weights) -- each
with R=4,096 replicas, 10 sweeps per temperature step, beta 0.1 -> 4.0 over
500 steps, adaptive reheating + NCM on, restart every 400 steps.  One timed
"step" is one iteration of Algorithm 1 (resample, NCM, 10 sweeps, energies,
M*, control) on BOTH instances.  attempts per step = R * N * S summed over the
two instances.  With K = 500 (the default) the timed steps are the whole
schedule of a fresh run.  With fewer, a pre-pass over the schedule (which is
also the warm-up; the controller's trajectory is fixed by the seed) finds the
iterations that apply cluster moves or reheat, and the K timed steps of a
fresh run are the window past step 40 (the stagnation windows are full from
there) that holds the most of them; the steps before the window run untimed.
The line also carries a "dense100k" object: the whole 200-step anneal of the
fully connected N=100,000 instance, device-timed, with its HBM roofline and
an end-to-end figure from host buffers.

Several GPUs (torchrun, one process per GPU): ONE population of R = 4,096 x
GPUs replicas per instance, split in equal blocks over the GPUs, with the
energies gathered and the migrating parent replicas exchanged by NCCL once
per iteration (weak scaling: 4,096 replicas per GPU and instance, as on one
GPU; the result equals the one-GPU run of the same R bit for bit).
--replicas runs independent populations instead; --split runs the split
path on one GPU (a group of one).

Timing: device time with CUDA events on the library's stream, one event pair
per step; between timed steps a 512 MB buffer is written to flush L2 (the
populations are smaller than L2).  The dominant kernel (the sweep) is also
timed on its own with events for the roofline line.

--impl reference runs the CPU oracle (the reference arm of this project: a
plain single-threaded C restatement of the paper) on a bounded sample of the
same workload.
"""
from __future__ import annotations

import argparse
import json
import os
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)
# The JSON lines go to JSON_OUT.  Run as a script, that is the process's
# original stdout and file descriptor 1 is pointed at stderr, so nothing else
# (NCCL's version banner, library messages) reaches stdout.
JSON_OUT = sys.stdout


def emit(obj) -> None:
    JSON_OUT.write(json.dumps(obj) + "\n")
    JSON_OUT.flush()


import workloads as W  # noqa: E402

R = 4096
SWEEPS = 10
STEPS_SCHEDULE = 500
PARAMS = dict(R=R, sweeps=SWEEPS, steps=STEPS_SCHEDULE, beta0=0.1, beta1=4.0, stagnation=1,
              z_rst=400, seed=0)
METRIC = "spin-flip attempts/s"
WORKLOAD = "augmented PAMC: torus 141x141 (+-1) + sparse N=7000 avg deg 5.7 (+-1), R=4096, 10 sweeps/step"


def load_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            return json.load(f), "measured"
    except OSError:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "sm_max_mhz": 2070.0}, "fallback"


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled during the timed region.

    One nvidia-smi process in loop mode (-lms) runs across the region; each
    sample carries nvidia-smi's own timestamp, and the summary keeps the
    samples that fall between the host times at which the region opened and
    closed.  The process is stopped with SIGINT (its normal end of loop mode),
    which flushes its output."""

    FIELDS = ("timestamp,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")
    REASONS = ("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap")
    INTERVAL_MS = 20
    WARM_IN_S = 0.5     # nvidia-smi start-up before the region opens

    def __init__(self, index: int = 0):
        self.index = index
        self.samples = []          # (unix time or None, [sm, max, power, 4 reasons])
        self.t0 = self.t1 = None
        self._proc = None
        self._started = 0.0

    @staticmethod
    def parse_line(line: str):
        import datetime
        f = [x.strip() for x in line.split(",")]
        if len(f) < 8:
            return None
        try:
            ts = datetime.datetime.strptime(f[0], "%Y/%m/%d %H:%M:%S.%f").timestamp()
        except ValueError:
            ts = None
        return ts, f[1:8]

    def start(self):
        """Start nvidia-smi ahead of the region (e.g. before the warm-up
        steps, so that its start-up does not leave the GPU idle)."""
        if self._proc is None:
            try:
                self._proc = subprocess.Popen(
                    ["nvidia-smi", "-i", str(self.index), "--query-gpu=" + self.FIELDS,
                     "--format=csv,noheader,nounits", "-lms", str(self.INTERVAL_MS)],
                    stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
                self._started = time.time()
            except OSError:
                self._proc = None
        return self

    def __enter__(self):
        self.start()
        if self._proc is not None:
            time.sleep(max(0.0, self.WARM_IN_S - (time.time() - self._started)))
        self.t0 = time.time()
        return self

    def __exit__(self, *a):
        import signal
        self.t1 = time.time()
        if self._proc is None:
            return
        try:
            time.sleep(2 * self.INTERVAL_MS / 1e3)   # one more sample after the region closes
            self._proc.send_signal(signal.SIGINT)
            out, _ = self._proc.communicate(timeout=10)
        except Exception:
            self._proc.kill()
            out, _ = self._proc.communicate()
        for line in (out or "").splitlines():
            r = self.parse_line(line)
            if r is not None:
                self.samples.append(r)

    def summary(self):
        inside = [f for ts, f in self.samples
                  if ts is not None and self.t0 is not None and self.t0 <= ts <= self.t1]
        window = "timed region"
        if not inside:
            # a region shorter than the sampling interval: the samples nearest to it
            near = sorted((abs(ts - (self.t0 + self.t1) / 2), f) for ts, f in self.samples if ts is not None)
            inside = [f for _, f in near[:2]] or [f for _, f in self.samples]
            window = "nearest to the timed region"
        if not inside:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"], "samples": 0}

        def num(x):
            try:
                return float(x)
            except ValueError:
                return None
        sm = [v for v in (num(f[0]) for f in inside) if v is not None]
        mx = [v for v in (num(f[1]) for f in inside) if v is not None]
        reasons = sorted({self.REASONS[i] for f in inside for i in range(4) if f[3 + i].lower() == "active"})
        return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "sm_mhz_min": min(sm) if sm else None, "reasons": reasons, "samples": len(inside),
                "window": window, "region_s": round(self.t1 - self.t0, 4)}


ONLY = None


def instances():
    insts = [W.c2a_torus141(), W.c2b_sparse7000()]
    if ONLY == "torus":
        return insts[:1]
    if ONLY == "sparse":
        return insts[1:]
    return insts


def attempts_per_step(insts):
    return sum(R * inst.n * SWEEPS for inst in insts)


# ---------------------------------------------------------------- reference arm
def run_reference(args):
    import oracle
    insts = instances()
    # bounded sample: the same instances and schedule, R_s replicas, one step each
    Rs = 32
    params = dict(PARAMS, R=Rs)

    def sample_step():
        att = 0
        for inst in insts:
            run = oracle.OracleRun(inst.row_ptr, inst.col, inst.w, **params)
            run.step(1)
            att += Rs * inst.n * SWEEPS
            run.close()
        return att

    for _ in range(args.warmup):     # untimed warm-up steps of the same sample
        sample_step()
    total_attempts = 0
    t_all = 0.0
    for k in range(args.steps):
        t0 = time.perf_counter()
        total_attempts += sample_step()
        t_all += time.perf_counter() - t0
    value = total_attempts / t_all
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": "attempts/s", "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * t_all / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "int32",
        "data": "synthetic", "config": {"workload": WORKLOAD, "R": R, "sweeps_per_step": SWEEPS,
                                        "sample": f"R={Rs} per instance, the first iteration of a run"},
        "cpu_baseline": {"value": value, "unit": "attempts/s", "cores": 1, "kind": "oracle",
                         "sample": f"first iteration of both instances with R={Rs} (same seeds)"},
        "e2e": {"value": value, "unit": "attempts/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    emit(line)


def cpu_baseline_sample():
    """Oracle timed on the host: first iteration of both instances, R=1024."""
    import oracle
    insts = instances()
    Rs = 1024
    params = dict(PARAMS, R=Rs)
    t0 = time.perf_counter()
    att = 0
    for inst in insts:
        run = oracle.OracleRun(inst.row_ptr, inst.col, inst.w, **params)
        run.step(1)
        att += Rs * inst.n * SWEEPS
        run.close()
    dt = time.perf_counter() - t0
    return {"value": att / dt, "unit": "attempts/s", "cores": 1, "kind": "oracle",
            "sample": f"first iteration (10 sweeps) of both instances with R={Rs}, {dt:.1f} s"}


# ---------------------------------------------------------------- our arm
def rank_seed(seed: int, rank: int) -> int:
    """Replicas only: rank r runs its own copy of the workload with seed + r."""
    return seed + rank


def reduce_over_ranks(dist, ms: float, attempts: float, device="cuda"):
    """Whole-job figures: the timed region is the max over ranks, the attempts
    the sum over ranks.  Returns (ms, attempts)."""
    if dist is None:
        return ms, attempts
    import torch
    t = torch.tensor([ms], dtype=torch.float64, device=device)
    a = torch.tensor([attempts], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    dist.all_reduce(a, op=dist.ReduceOp.SUM)
    return float(t.item()), float(a.item())


def run_ours(args):
    import torch
    import paper_2606_25203_gb300 as pg

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dist = None
    if world > 1 or args.split:
        import torch.distributed as dist
        if world == 1 and "MASTER_ADDR" not in os.environ:
            os.environ.setdefault("MASTER_ADDR", "127.0.0.1")
            os.environ.setdefault("MASTER_PORT", "29541")
            os.environ.setdefault("RANK", "0")
        dist.init_process_group("nccl", world_size=world, rank=rank)
    pg.load()
    if (world > 1 and not args.replicas) or args.split:
        return run_split(args, pg, torch, dist, rank, world, local)
    insts = instances()
    stream = torch.cuda.current_stream()
    # the two instances are independent: each steps on a stream of its own
    # (unless --one-stream), so one's kernels fill the other's last wave
    sstreams = [stream if args.one_stream else torch.cuda.Stream() for _ in insts]
    solvers = []
    for inst, st in zip(insts, sstreams):
        s = pg.Solver(inst.row_ptr, inst.col, inst.w, device=local, stream=st.cuda_stream)
        s.init(**dict(PARAMS, seed=rank_seed(PARAMS["seed"], rank)))
        solvers.append(s)
    flush = torch.empty(512 * 1024 * 1024 // 4, dtype=torch.int32, device="cuda")
    clk = ClockSampler(local).start()
    run_params = dict(PARAMS, seed=rank_seed(PARAMS["seed"], rank))
    # the work of a step depends on where it is in the schedule (control,
    # cluster moves, restart): place the timed window
    if args.steps >= STEPS_SCHEDULE or args.lean:      # profiling runs time steps 0..K-1
        for _ in range(args.warmup):
            for s in solvers:
                s.step(1)
        start, events = 0, None
    else:
        events = schedule_events(solvers)          # also the warm-up
        start = choose_window(events, args.steps)
    for s in solvers:
        s.init(**run_params)
        s.step(start)                              # untimed steps before the window
        pg.pamc_set_sweep_timing(s.h, True)
    torch.cuda.synchronize()
    sw0 = [pg.pamc_sweep_stats(s.h) for s in solvers]   # resets the sweep timers
    ctl0 = [s.control() for s in solvers]
    launches0 = sum(s.launches() for s in solvers)
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
          for _ in range(args.steps)]
    done = [torch.cuda.Event() for _ in solvers]
    with clk:
        for k in range(args.steps):
            flush.add_(1)
            ev[k][0].record(stream)
            for s, st, d in zip(solvers, sstreams, done):
                st.wait_event(ev[k][0])          # the step starts after the flush
                s.step(1)
                d.record(st)
            for d in done:
                stream.wait_event(d)             # and ends when both instances' iterations have
            ev[k][1].record(stream)
        torch.cuda.synchronize()
    if dist:
        dist.barrier()
    launches = sum(s.launches() for s in solvers) - launches0
    ms = sum(a.elapsed_time(b) for a, b in ev)
    for s in solvers:
        s.sync()
    ctl1 = [s.control() for s in solvers]
    sw1 = [pg.pamc_sweep_stats(s.h) for s in solvers]
    for s in solvers:
        pg.pamc_set_sweep_timing(s.h, False)
    window = window_summary(events, start, args.steps, ctl0, ctl1)
    ms, att = reduce_over_ranks(dist, ms, attempts_per_step(insts) * args.steps)
    value = att / (ms / 1e3)

    if args.lean:
        if rank == 0:
            emit({"metric": METRIC, "value": value, "unit": "attempts/s",
                              "ms_per_step": ms / args.steps, "gpu_launches": launches,
                              "clocks": clk.summary(), "config": {"only": ONLY}})
        for s in solvers:
            s.close()
        return None
    # dominant kernel: the sweep launches of the timed window, each timed by
    # CUDA events the library records around it on its stream
    peaks, peak_src = load_peaks()
    sm_max = peaks.get("sm_max_mhz", 2070.0)
    sweep = [sweep_roofline(inst, args.steps, a, b, sm_max) for inst, a, b in zip(insts, sw0, sw1)]
    # the same kernel without the other instance's launches beside it: the K
    # steps after the window, the first instance alone on its stream
    pg.pamc_set_sweep_timing(solvers[0].h, True)
    torch.cuda.synchronize()
    iso0 = pg.pamc_sweep_stats(solvers[0].h)
    for _ in range(args.steps):
        solvers[0].step(1)
    solvers[0].sync()
    iso = sweep_roofline(insts[0], args.steps, iso0, pg.pamc_sweep_stats(solvers[0].h), sm_max)
    pg.pamc_set_sweep_timing(solvers[0].h, False)
    mode = [pg.pamc_sweep_mode(s.h) for s in solvers]
    kname = ["k_sweep_ising_bits" if m & 32 else "k_sweep_ising_nib" if m & 16 else "k_sweep_ising_push" if m == 2 else "k_sweep_ising" for m in mode]
    e2e = e2e_measure(pg, torch, insts, args, local, start)
    dense = None
    if world == 1 and not args.no_dense:
        for s in solvers:
            s.close()
        solvers = []
        torch.cuda.empty_cache()
        dense = dense_measure(pg, torch, DENSE_N, DENSE_PARAMS["steps"], args.warmup, e2e=True)
    result = None
    if rank == 0:
        cpu = cpu_baseline_sample() if world == 1 else None
        result = {
            "metric": METRIC, "value": value, "unit": "attempts/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "int32", "data": "synthetic",
            "config": {"workload": WORKLOAD, "R": R, "sweeps_per_step": SWEEPS,
                       "attempts_per_step": attempts_per_step(insts), "l2": "flushed between steps (512 MB write)",
                       "timed_steps": f"steps {start}..{start + args.steps - 1} of a fresh run "
                                      f"({STEPS_SCHEDULE}-step schedule, restart every {PARAMS['z_rst']}"
                                      + (f"; steps 0..{start - 1} untimed" if start else "") + ")",
                       "timed_window": window,
                       "parallelism": "replicas only" if world > 1 else "single GPU"},
            "roofline": dict(sweep[0], traffic=None,
                             kernel=kname[0] + f" ({insts[0].name}, R=4096, 10 sweeps per launch)",
                             peak_source=f"152 SMs x 128 int32 lanes x {sm_max:.0f} MHz ({peak_src} clock)",
                             note="launches of the timed window, beside the other instance's on their own stream "
                                  "(the SMs are shared, so each launch is stretched)",
                             alone={k: iso[k] for k in ("achieved", "frac", "avg_launch_ms", "launches",
                                                        "pull_count")}
                                   | {"window": f"steps {start + args.steps}..{start + 2 * args.steps - 1}, "
                                                f"this instance alone"}),
            "clocks": clk.summary(),
            "gpu_launches": launches,
            "e2e": e2e,
            "cpu_baseline": cpu,
            "dense100k": dense,
        }
        emit(result)
    for s in solvers:
        s.close()
    if dist:
        dist.destroy_process_group()
    return result


R_MAX = 1 << 20   # the largest population pamc_init takes


def split_groups(world: int) -> int:
    """GPUs per population: the largest divisor of world whose population of
    4,096 replicas per GPU pamc_init takes (R <= 1,048,576): all of them up
    to 256 GPUs."""
    return max(d for d in range(1, world + 1) if world % d == 0 and d * R <= R_MAX)


def run_split(args, pg, torch, dist, rank, world, local):
    """Several GPUs: ONE population of R = 4,096 x GPUs replicas per instance
    (several of at most 1,048,576 beyond 256 GPUs), split in equal blocks over
    the GPUs (weak scaling: every GPU sweeps 4,096 replicas of each instance,
    as on one GPU).  Every
    iteration gathers the R energies of a population (NCCL all-gather), runs
    the same population step and controller on each of its GPUs, and moves
    the parent replicas that live on another GPU (NCCL all-to-all); the
    result equals the one-GPU run of the same R bit for bit.  The timed
    steps are the iterations the one-GPU line times (its pre-pass on one
    GPU's population picks them)."""
    from paper_2606_25203_gb300 import shard as S
    insts = instances()
    G = split_groups(world)
    npop = world // G
    pop, prank = rank // G, rank % G
    groups = [dist.new_group(list(range(q * G, (q + 1) * G))) for q in range(npop)] if npop > 1 else [None]
    Rg = R * G
    params = dict(PARAMS, R=Rg, seed=PARAMS["seed"] + pop)
    comm = S.TorchComm(groups[pop])
    streams = [torch.cuda.Stream() for _ in insts]
    start, events = 0, None
    if args.steps < STEPS_SCHEDULE and not args.lean:
        probe = [pg.Solver(inst.row_ptr, inst.col, inst.w, device=local) for inst in insts]
        for s in probe:
            s.init(**PARAMS)
        events = schedule_events(probe)
        start = choose_window(events, args.steps)
        for s in probe:
            s.close()

    def make():
        out = []
        for inst, st in zip(insts, streams):
            with torch.cuda.stream(st):
                out.append(S.LibShard(inst.row_ptr, inst.col, inst.w, prank, G, device=local, **params))
        return out

    def step_all(shards):
        for sh, st in zip(shards, streams):
            with torch.cuda.stream(st):
                S.run_step(sh, comm)

    if start < args.warmup:              # warm-up on a population of its own
        warm = make()
        for _ in range(args.warmup):
            step_all(warm)
        for sh in warm:
            sh.close()
    shards = make()
    for _ in range(start):               # untimed iterations before the window
        step_all(shards)
    for sh in shards:
        pg.pamc_set_sweep_timing(sh.h, True)
    torch.cuda.synchronize()
    sw0 = [pg.pamc_sweep_stats(sh.h) for sh in shards]
    ctl0 = [pg.pamc_control_state(sh.h) for sh in shards]
    launches0 = sum(pg.pamc_launch_count(sh.h) for sh in shards)
    moved0 = sum(sh.moved for sh in shards)
    flush = torch.empty(512 * 1024 * 1024 // 4, dtype=torch.int32, device="cuda")
    clk = ClockSampler(local).start()
    cur = torch.cuda.current_stream()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
          for _ in range(args.steps)]
    dist.barrier()
    torch.cuda.synchronize()
    with clk:
        for k in range(args.steps):
            flush.add_(1)
            ev[k][0].record(cur)
            for st in streams:
                st.wait_stream(cur)
            step_all(shards)
            for st in streams:
                cur.wait_stream(st)
            ev[k][1].record(cur)
        torch.cuda.synchronize()
    dist.barrier()
    ms = sum(a.elapsed_time(b) for a, b in ev)
    launches = sum(pg.pamc_launch_count(sh.h) for sh in shards) - launches0
    moved = sum(sh.moved for sh in shards) - moved0
    ctl1 = [pg.pamc_control_state(sh.h) for sh in shards]
    sw1 = [pg.pamc_sweep_stats(sh.h) for sh in shards]
    own_attempts = sum(sh.count * inst.n * SWEEPS for sh, inst in zip(shards, insts)) * args.steps
    ms, att = reduce_over_ranks(dist, ms, own_attempts)
    value = att / (ms / 1e3)
    for sh in shards:
        pg.pamc_set_sweep_timing(sh.h, False)
        sh.close()
    if args.lean:
        if rank == 0:
            emit({"metric": METRIC, "value": value, "unit": "attempts/s", "n_gpus": world,
                              "ms_per_step": ms / args.steps, "gpu_launches": launches, "clocks": clk.summary(),
                              "config": {"only": ONLY, "R_total": Rg, "populations": npop, "split": True}})
        dist.destroy_process_group()
        return None
    peaks, peak_src = load_peaks()
    sm_max = peaks.get("sm_max_mhz", 2070.0)
    sweep = sweep_roofline(insts[0], args.steps, sw0[0], sw1[0], sm_max)
    e2e = split_e2e(args, pg, torch, S, comm, insts, params, prank, G, local, start, dist)
    result = None
    if rank == 0:
        result = {
            "metric": METRIC, "value": value, "unit": "attempts/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "int32", "data": "synthetic",
            "config": {"workload": WORKLOAD.replace("R=4096", f"{npop} population(s) of R={Rg} per instance"),
                       "R": Rg, "populations": npop, "gpus_per_population": G, "R_per_gpu": R,
                       "sweeps_per_step": SWEEPS,
                       "attempts_per_step": attempts_per_step(insts) * world,
                       "l2": "flushed between steps (512 MB write)",
                       "timed_steps": f"steps {start}..{start + args.steps - 1} of a fresh run",
                       "timed_window": window_summary(events, start, args.steps, ctl0, ctl1),
                       "parallelism": f"{npop} population(s), each split over {G} GPU(s): replica blocks, NCCL "
                                      f"all-gather of the energies and all-to-all of the migrating replicas per "
                                      f"iteration",
                       "replicas_moved_per_step": moved / args.steps},
            "roofline": dict(sweep, traffic=None,
                             kernel=f"k_sweep_ising ({insts[0].name}, 4096 replicas per GPU, 10 sweeps per launch)",
                             peak_source=f"152 SMs x 128 int32 lanes x {sm_max:.0f} MHz ({peak_src} clock)"),
            "clocks": clk.summary(),
            "gpu_launches": launches,
            "e2e": e2e,
            "cpu_baseline": None,
        }
        emit(result)
    dist.destroy_process_group()
    return result


def split_e2e(args, pg, torch, S, comm, insts, params, rank, world, local, start, dist):
    """End to end through the public API with host buffers, for the split
    population: each process uploads the instance (host CSR) and draws its
    block, runs the iterations up to the end of the window, and after every
    iteration the best cut and its configuration reach every process's host
    (the holder broadcasts it); all of it timed, max over processes."""
    streams = [torch.cuda.Stream() for _ in insts]
    dist.barrier()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    h2d = d2h = 0
    shards = []
    for inst, st in zip(insts, streams):
        with torch.cuda.stream(st):
            shards.append(S.LibShard(inst.row_ptr, inst.col, inst.w, rank, world, device=local, **params))
        h2d += inst.row_ptr.nbytes + inst.col.nbytes + inst.w.nbytes
    nsteps = start + args.steps
    for _ in range(nsteps):
        for sh, st in zip(shards, streams):
            with torch.cuda.stream(st):
                S.run_step(sh, comm)
        for sh, st in zip(shards, streams):
            with torch.cuda.stream(st):
                S.best(sh, comm)
            d2h += 8 + sh.n
    torch.cuda.synchronize()
    dt = time.perf_counter() - t0
    for sh in shards:
        sh.close()
    own = sum(sh.count * inst.n * SWEEPS for sh, inst in zip(shards, insts)) * nsteps
    ms, att = reduce_over_ranks(dist, dt * 1e3, own)
    return {"value": att / (ms / 1e3), "unit": "attempts/s", "h2d_bytes_per_step": h2d / nsteps,
            "d2h_bytes_per_step": d2h / nsteps, "steps": nsteps}


def schedule_events(solvers):
    """One pass over the whole schedule of each run, reading the controller
    after every iteration: the iterations that applied cluster moves, that
    reheated (strong stagnation: the cluster move armed), and that restarted.
    The trajectory is a function of the seed, so a fresh run with the same
    seed meets the same events at the same steps."""
    ev = []
    for s in solvers:
        ncm, reheat, restart = [], [], []
        prev = s.control()
        for t in range(STEPS_SCHEDULE):
            s.step(1)
            c = s.control()
            if c["ncm_last"]:
                ncm.append(t)
            if c["enable_cm"] and not prev["enable_cm"]:
                reheat.append(t)
            if c["cycle"] > prev["cycle"]:
                restart.append(t)
            prev = c
        ev.append({"ncm": ncm, "reheat": reheat, "restart": restart})
    return ev


def choose_window(events, K, lo=40):
    """First step of the K-step window at or after lo (the stagnation windows
    hold 40 values from there) that contains the most cluster-move and reheat
    iterations of all runs; ties to the earliest."""
    hi = max(lo, STEPS_SCHEDULE - K)
    marks = sorted(t for e in events for t in e["ncm"] + e["reheat"])
    best, best_n = lo, -1
    for a in range(lo, hi + 1):
        n = sum(1 for t in marks if a <= t < a + K)
        if n > best_n:
            best, best_n = a, n
    return best


def window_summary(events, start, K, ctl0, ctl1):
    """What the timed window contains: from the pre-pass, the iterations of
    each run that applied cluster moves, reheated or restarted; from the
    timed run itself, the spins the cluster moves flipped in the window."""
    out = {"first": start, "last": start + K - 1,
           "ncm_spins_flipped": [int(b["ncm_flipped"] - a["ncm_flipped"]) for a, b in zip(ctl0, ctl1)]}
    if events is not None:
        for key in ("ncm", "reheat", "restart"):
            out[key + "_steps"] = [[t for t in e[key] if start <= t < start + K] for e in events]
    return out


# Algorithmic 32-bit integer operations of the sweeps (Eq. 3-4 with
# incrementally kept fields): per spin-flip attempt a quarter of one
# Philox4x32-10 call (10 rounds x 6 ops: 2 mul-hi, 2 mul-lo, 2 three-way xor)
# and 3 for the threshold (index, load, compare); per accepted flip 1 for the
# spin and 2 per incident coupling (read-modify-write of the neighbour field).
OPS_PER_ATTEMPT = 60 / 4 + 3


def ops_per_flip(inst):
    return 1 + 2 * inst.nnz / inst.n


def sweep_roofline(inst, steps, before, after, sm_max):
    """ALU roofline of one instance's sweep launches in the timed window:
    algorithmic operations (attempts and counted flips) over their summed
    event time (each launch timed by the library on its stream)."""
    att = R * inst.n * SWEEPS * steps
    flips = after["flips"] - before["flips"]
    ops = att * OPS_PER_ATTEMPT + flips * ops_per_flip(inst)
    ms, launches = after["ms"], after["launches"]
    achieved = ops / (ms / 1e3) / 1e12
    peak = 152 * 128 * sm_max * 1e6 / 1e12
    # the same launches on the pull sweep's own count (every attempt reads its
    # neighbours: 2 ops per incident coupling, no flip term), the count of
    # earlier figures, for comparison
    pull_ops = OPS_PER_ATTEMPT + 2.0 * inst.nnz / inst.n
    pull_frac = att * pull_ops / (ms / 1e3) / 1e12 / peak
    return {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "Tops/s", "frac": achieved / peak,
            "launches": launches, "avg_launch_ms": ms / max(launches, 1), "sweep_ms": ms,
            "ops_per_attempt": OPS_PER_ATTEMPT, "ops_per_flip": ops_per_flip(inst),
            "flip_fraction": flips / att, "attempts_per_s": att / (ms / 1e3),
            "pull_count": {"ops_per_attempt": pull_ops, "frac": pull_frac}}


def e2e_measure(pg, torch, insts, args, device, start=0):
    """End to end through the public API with host buffers: instance upload
    (host CSR -> device), init, the untimed steps before the window and the K
    window iterations, each iteration followed by a read of the best cut and
    configuration to the host; all of it inside the timed region, and the
    attempts of every step run counted."""
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    h2d = 0
    d2h = 0
    solvers = []
    streams = [None if args.one_stream else torch.cuda.Stream() for _ in insts]
    for inst, st in zip(insts, streams):
        s = pg.Solver(inst.row_ptr, inst.col, inst.w, device=device,
                      stream=None if st is None else st.cuda_stream)
        h2d += inst.row_ptr.nbytes + inst.col.nbytes + inst.w.nbytes
        s.init(**PARAMS)
        solvers.append(s)
    nsteps = start + args.steps
    for _ in range(nsteps):
        for s in solvers:          # both instances' iterations enqueued, then both read back
            s.step(1)
        for s in solvers:
            s.best()
            d2h += 8 + s.n
    torch.cuda.synchronize()
    dt = time.perf_counter() - t0
    for s in solvers:
        s.close()
    att = attempts_per_step(insts) * nsteps
    return {"value": att / dt, "unit": "attempts/s", "h2d_bytes_per_step": h2d / nsteps,
            "d2h_bytes_per_step": d2h / nsteps, "steps": nsteps}


# ---------------------------------------------------------------- dense 100k
DENSE_N = 100_000
DENSE_PARAMS = dict(R=64, sweeps=2, steps=200, beta0=0.01, beta1=1.0, stagnation=0, seed=0)
DENSE_WORKLOAD = "fully connected Ising N=100,000, J=+-1 dense int8 (10 GB), R=64, 2 sweeps/step"


def dense_weights_device(torch, n, seed=0, chunk=2000):
    """Max-Cut weights w = -J of the dense +-1 instance, built on the device."""
    w = torch.empty((n, n), dtype=torch.int8, device="cuda")
    for r0 in range(0, n, chunk):
        r1 = min(n, r0 + chunk)
        w[r0:r1] = -W.dense_rows_torch(n, r0, r1, seed, device="cuda")
    return w


def dense_measure(pg, torch, n, steps, warmup, e2e=False):
    """Configuration 4: steps 0..steps-1 of a fresh anneal of the dense
    instance, device-timed step by step (the instance, 10 GB at n = 100,000,
    is larger than L2), the kernel split (a step without sweeps), the HBM
    roofline of the sweep (one read of J per sweep) and of the recompute (one
    read of J per step), and the rows the flips needed.  With e2e, the same
    steps again through the public API from a host copy of the weights:
    upload, validation, init, every step followed by a read of the best cut
    and configuration, all inside the wall-clock region."""
    stream = torch.cuda.current_stream()
    t0 = time.perf_counter()
    w = dense_weights_device(torch, n)
    torch.cuda.synchronize()
    gen_s = time.perf_counter() - t0
    w_host = None
    if e2e:   # the weights in pinned host memory, as a caller streaming instances would hold them
        w_pin = torch.empty((n, n), dtype=torch.int8, pin_memory=True)
        w_pin.copy_(w)
        w_host = w_pin.numpy()
    h = pg.pamc_create_dense(n, w, stream=stream.cuda_stream)
    del w
    torch.cuda.empty_cache()
    P = dict(DENSE_PARAMS)
    # warm-up steps on a throwaway run, then the timed steps 0..K-1 of a fresh
    # run (the cost of a step depends on where it is in the beta schedule)
    pg.pamc_init(h, **P)
    pg.pamc_step(h, warmup)
    pg.pamc_sync(h)
    pg.pamc_init(h, **P)
    pg.pamc_set_sweep_timing(h, True)
    torch.cuda.synchronize()
    pg.pamc_sweep_stats(h)                       # resets the sweep timers
    l0 = pg.pamc_launch_count(h)
    rows0, pos0 = pg.pamc_dense_rows(h)
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
          for _ in range(steps)]
    with ClockSampler(0) as clk:
        for k in range(steps):
            ev[k][0].record(stream)
            pg.pamc_step(h, 1)
            ev[k][1].record(stream)
        torch.cuda.synchronize()
    pg.pamc_sync(h)
    sw = pg.pamc_sweep_stats(h)                  # the sweep launches of the timed steps
    pg.pamc_set_sweep_timing(h, False)
    rows1, pos1 = pg.pamc_dense_rows(h)
    per_step = [a.elapsed_time(b) for a, b in ev]
    ms = sum(per_step)
    launches = pg.pamc_launch_count(h) - l0
    att = P["R"] * n * P["sweeps"] * steps
    m, _ = pg.pamc_best(h, n)
    e_best = pg.pamc_weight_sum(h) - 2 * m     # E = W - 2 cut
    # kernel split: a step without sweeps (order, resampling, tables, the
    # tensor-core recompute, control) on the same population
    pg.pamc_init(h, **dict(P, sweeps=0))
    pg.pamc_step(h, 2)
    torch.cuda.synchronize()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record(stream)
    pg.pamc_step(h, 3)
    b.record(stream)
    torch.cuda.synchronize()
    ms_nosweep = a.elapsed_time(b) / 3
    ms_sweep = sw["ms"] / max(sw["launches"], 1)   # one sweep launch per step
    pg.pamc_destroy(h)
    peaks, src = load_peaks()
    hbm = peaks["hbm_gbs"]
    rc_gbs = n * n / 8 / (ms_nosweep / 1e3) / 1e9            # J (one bit a coupling) of the recompute
    sw_gbs = P["sweeps"] * n * n / 8 / (ms_sweep / 1e3) / 1e9  # one read of J per sweep
    e2e_obj = None
    if e2e:
        torch.cuda.synchronize()
        t1 = time.perf_counter()
        h = pg.pamc_create_dense(n, w_host, stream=stream.cuda_stream)
        pg.pamc_init(h, **P)
        for _ in range(steps):
            pg.pamc_step(h, 1)
            pg.pamc_best(h, n)
        dt = time.perf_counter() - t1
        pg.pamc_destroy(h)
        e2e_obj = {"value": att / dt, "unit": "attempts/s", "h2d_bytes_per_step": n * n / steps,
                   "d2h_bytes_per_step": 8 + n, "steps": steps,
                   "includes": "upload of the n x n weights from pinned host memory, validation, init"}
    del w_host
    if e2e:
        del w_pin
    return {
        "metric": METRIC, "value": att / (ms / 1e3), "unit": "attempts/s", "n_gpus": 1,
        "steps": steps, "warmup": warmup, "ms_per_step": ms / steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "int32",
        "data": "synthetic", "config": {"workload": DENSE_WORKLOAD, "n": n, **P,
                                        "l2": "inputs (1.25 GB of coupling bits) larger than L2"},
        "kernels_ms": {"step": ms / steps, "sweeps": ms_sweep, "sweep_launches_timed": sw["launches"],
                       "step_without_sweeps": ms_nosweep},
        "roofline": {"bound": "hbm", "achieved": sw_gbs, "peak": hbm, "unit": "GB/s",
                     "frac": sw_gbs / hbm,
                     "traffic": None,
                     "kernel": "k_dense_sweep (bytes = one read of J, one bit a coupling, per sweep)",
                     "peak_source": src},
        # (what bounds the recompute is the way of its operands into tensor memory)
        "recompute_roofline": {"bound": "tensor memory", "achieved": rc_gbs, "peak": hbm, "unit": "GB/s",
                               "frac": rc_gbs / hbm},
        # the rows the flips needed: positions that flipped in at least one
        # replica; their rows (n bits each) are all a sweep's field updates read of J
        "rows_needed": {"rows": rows1 - rows0, "positions": pos1 - pos0,
                        "fraction": (rows1 - rows0) / max(pos1 - pos0, 1),
                        "achieved_gbs": (rows1 - rows0) * n / 8 / (ms_sweep * steps / 1e3) / 1e9},
        "e2e": e2e_obj,
        "clocks": clk.summary(), "gpu_launches": launches,
        "timed_steps": f"steps 0..{steps - 1} of a fresh run (beta {P['beta0']} -> {P['beta1']} over {P['steps']})",
        "ms_step_first_last": [per_step[0], per_step[-1]],
        # where the anneal's time goes: mean step time over windows of 10 steps
        "ms_step_windows": {"size": 10, "mean_ms": [round(sum(per_step[i:i + 10]) / len(per_step[i:i + 10]), 3)
                                                     for i in range(0, len(per_step), 10)]},
        "best_cut": m, "best_energy_density": e_best / n ** 1.5,
        "instance_generation_s": gen_s,
    }


def run_dense(args):
    import torch
    import paper_2606_25203_gb300 as pg
    world = int(os.environ.get("WORLD_SIZE", "1"))
    if world > 1 or args.split:
        return run_dense_split(args, pg, torch, world)
    pg.load()
    emit(dense_measure(pg, torch, args.dense_n, args.steps, args.warmup, e2e=args.dense_e2e))


def run_dense_split(args, pg, torch, world):
    """Configuration 4 on several GPUs: one population of R = 64 x GPUs,
    64 replicas per GPU (weak scaling), J on every GPU; every iteration
    gathers the energies, runs the same population step everywhere and moves
    the parent replicas (n int8 each) that live on another GPU (NCCL).
    Steps 0..K-1 of a fresh anneal (after K warm-up steps of another run),
    device-timed, max over GPUs."""
    import torch.distributed as dist
    from paper_2606_25203_gb300 import shard as S
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    if world == 1 and "MASTER_ADDR" not in os.environ:
        os.environ.setdefault("MASTER_ADDR", "127.0.0.1")
        os.environ.setdefault("MASTER_PORT", "29543")
    dist.init_process_group("nccl", world_size=world, rank=rank)
    pg.load()
    n = args.dense_n
    w = dense_weights_device(torch, n)
    params = dict(DENSE_PARAMS, R=64 * world)
    comm = S.TorchComm()
    cur = torch.cuda.current_stream()

    def make():
        return S.LibShard(None, None, None, rank, world, device=local, dense_w=w, **params)

    warm = make()
    for _ in range(args.warmup):
        S.run_step(warm, comm)
    warm.close()
    sh = make()
    del w
    torch.cuda.empty_cache()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    dist.barrier()
    torch.cuda.synchronize()
    with ClockSampler(local) as clk:
        for k in range(args.steps):
            ev[k][0].record(cur)
            S.run_step(sh, comm)
            ev[k][1].record(cur)
        torch.cuda.synchronize()
    dist.barrier()
    ms = sum(a.elapsed_time(b) for a, b in ev)
    own = sh.count * n * params["sweeps"] * args.steps
    ms, att = reduce_over_ranks(dist, ms, own)
    cut, _ = S.best(sh, comm)
    moved = sh.moved
    sh.close()
    if rank == 0:
        emit({
            "metric": METRIC, "value": att / (ms / 1e3), "unit": "attempts/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "int32", "data": "synthetic",
            "config": {"workload": DENSE_WORKLOAD.replace("R=64", f"one population of R={64 * world}"),
                       "n": n, "R": 64 * world, "R_per_gpu": 64,
                       "parallelism": f"one population split over {world} GPU(s), NCCL exchange per iteration",
                       "replicas_moved_per_step": moved / args.steps,
                       "timed_steps": f"steps 0..{args.steps - 1} of a fresh run"},
            "best_cut": int(cut), "clocks": clk.summary()})
    dist.destroy_process_group()


SERVE_PARAMS = dict(R=512, sweeps=10, steps=200, beta0=0.1, beta1=3.0, seed=0)
SERVE_WORKLOAD = ("serving stream: Max-Cut and Max-3-Cut requests, N ~ U[800, 20000], ER unit / ER +-1 "
                  "(avg deg 20) / torus +-1, R=512, 200 steps x 10 sweeps each")


def run_serving(args):
    """Continuous batching against one-instance-per-launch on the same requests.

    Throughput: a saturating stream (all requests present at t=0) served by the
    batched loop and by the plain path, solves/s = requests / makespan (host
    wall clock, instances uploaded from host memory and best cuts read back
    inside the region).  Latency: a second batched pass with Poisson arrivals
    at half the measured batched capacity, p50/p99 of (finish - arrival)."""
    import torch
    import paper_2606_25203_gb300 as pg
    from paper_2606_25203_gb300.serving import Server, serve_sequential
    pg.load()
    P = dict(SERVE_PARAMS)
    nreq = args.serve_requests
    t0 = time.perf_counter()
    burst = W.serving_stream(nreq, rate=0.0, seed=1, max3cut_frac=args.serve_max3cut)
    gen_s = time.perf_counter() - t0
    warm = W.serving_stream(max(3, args.warmup), rate=0.0, seed=2, n_lo=800, n_hi=2000)
    wp = dict(P, steps=4)
    srv = Server(max_active=args.serve_max_active, steps_per_tick=2)
    # launch shape per size class, tuned on copies of requests from another stream
    t1 = time.perf_counter()
    tune_reqs = W.serving_stream(24, rate=0.0, seed=3, max3cut_frac=args.serve_max3cut)
    samples = []
    for lo, hi in ((800, 2048), (2049, 8192), (8193, 20000)):
        samples += [(r.inst, r.kind) for r in tune_reqs if lo <= r.inst.n <= hi][:6]
    shapes = srv.autotune(samples, P)
    tune_s = time.perf_counter() - t1
    srv.serve(warm, wp)
    serve_sequential(warm, wp)
    torch.cuda.synchronize()
    attempts = sum(P["R"] * r.inst.n * P["sweeps"] * P["steps"] for r in burst)
    with ClockSampler(0) as clk:
        st = srv.serve(burst, P)
        torch.cuda.synchronize()
    seq = serve_sequential(burst, P)
    cuts = {r.rid: r.cut for r in seq.results}
    identical = all(cuts[r.rid] == r.cut for r in st.results) and len(st.results) == nreq
    cap = st.solves_per_s
    poisson = W.serving_stream(nreq, rate=0.5 * cap, seed=1, max3cut_frac=args.serve_max3cut)
    lt = srv.serve(poisson, P)
    srv.close()
    peaks, src = load_peaks()
    sm_max = peaks.get("sm_max_mhz", 2070.0)
    alu_peak = 152 * 128 * sm_max * 1e6 / 1e9   # Gop/s of 32-bit ALU lanes
    ops = sum(P["R"] * r.inst.n * P["sweeps"] * P["steps"] * (18 + 2 * r.inst.nnz / r.inst.n) for r in burst)
    ach = ops / st.makespan / 1e9
    line = {
        "metric": "batched solves/s", "value": cap, "unit": "solves/s", "n_gpus": 1,
        "steps": nreq, "warmup": len(warm), "ms_per_step": st.makespan / nreq * 1e3,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "int32",
        "data": "synthetic",
        "config": {"workload": SERVE_WORKLOAD, "requests": nreq, "max3cut_requests": sum(r.kind for r in burst),
                   **P, "max_active": args.serve_max_active,
                   "timing": "host wall clock over the whole stream (upload, init, steps, best-cut readback)",
                   "l2": "populations and schedule rings of the resident requests exceed L2"},
        "p50_s": lt.latency_pct(50), "p99_s": lt.latency_pct(99),
        "latency_load": {"rate_per_s": 0.5 * cap, "solves_per_s": lt.solves_per_s},
        "burst_p50_s": st.latency_pct(50), "burst_p99_s": st.latency_pct(99),
        "one_instance_per_launch": {"value": seq.solves_per_s, "unit": "solves/s",
                                    "p50_s": seq.latency_pct(50), "p99_s": seq.latency_pct(99),
                                    "gpu_launches": seq.launches},
        "speedup_vs_one_instance_per_launch": cap / seq.solves_per_s if seq.solves_per_s else None,
        "identical_cuts": identical,
        "attempts_per_s": attempts / st.makespan,
        "roofline": {"bound": "alu", "achieved": ach, "peak": alu_peak, "unit": "Gop/s", "frac": ach / alu_peak,
                     "traffic": None, "kernel": "whole batched stream (all kernels, host gaps included)",
                     "peak_source": "152 SMs x 128 int32 lanes x max SM clock"},
        "e2e": {"value": cap, "unit": "solves/s",
                "h2d_bytes_per_step": int(np.mean([4 * (r.inst.n + 1) + 8 * r.inst.nnz for r in burst])),
                "d2h_bytes_per_step": int(np.mean([r.inst.n + 8 for r in burst]))},
        "clocks": clk.summary(), "gpu_launches": st.launches, "graph_builds": st.graph_builds,
        "peak_active": st.peak_active, "peak_resident_bytes": st.peak_bytes,
        "batch_shapes": {str(c): {"groups_per_cta": g, "warps_per_group": w, "lanes_per_vertex": lv,
                                  "spins_in_device_memory": bool(gm), "ms_per_step": ms}
                         for c, (g, w, lv, ms, gm) in shapes.items()},
        "autotune_s": tune_s,
        "request_generation_s": gen_s,
    }
    emit(line)


def run_batch(args):
    """A fixed batch of serving requests resident on the device, advanced by
    pamc_batch_step: device-timed steps (CUDA events on the batch stream), the
    throughput of the batched kernels without admission or host gaps."""
    import torch
    import paper_2606_25203_gb300 as pg
    pg.load()
    P = dict(SERVE_PARAMS, steps=1 << 20)
    reqs = W.serving_stream(args.batch_requests, rate=0.0, seed=1, n_lo=args.batch_n_lo, n_hi=args.batch_n_hi)
    st = torch.cuda.Stream()
    b = pg.pamc_batch_create(0, st.cuda_stream)
    hs = []
    for r in reqs:
        h = pg.pamc_create_csr(r.inst.n, r.inst.row_ptr, r.inst.col, r.inst.w, 0, st.cuda_stream)
        pg.pamc_init(h, **P)
        pg.pamc_batch_add(b, h)
        hs.append(h)
    pg.pamc_batch_step(b, args.warmup)
    torch.cuda.synchronize()
    l0 = pg.pamc_batch_launch_count(b)
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    with ClockSampler(0) as clk:
        for k in range(args.steps):
            ev[k][0].record(st)
            pg.pamc_batch_step(b, 1)
            ev[k][1].record(st)
        torch.cuda.synchronize()
    ms = sum(a.elapsed_time(c) for a, c in ev)
    att = sum(P["R"] * r.inst.n * P["sweeps"] for r in reqs) * args.steps
    ops = sum(P["R"] * r.inst.n * P["sweeps"] * (18 + 2 * r.inst.nnz / r.inst.n) for r in reqs) * args.steps
    peaks, src = load_peaks()
    alu_peak = 152 * 128 * peaks.get("sm_max_mhz", 2070.0) * 1e6 / 1e12
    ach = ops / (ms / 1e3) / 1e12
    line = {
        "metric": METRIC, "value": att / (ms / 1e3), "unit": "attempts/s", "n_gpus": 1, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "int32", "data": "synthetic",
        "config": {"workload": f"batch of {len(reqs)} resident serving requests, N ~ U[{args.batch_n_lo}, "
                               f"{args.batch_n_hi}], R=512, 10 sweeps/step",
                   "l2": "populations and schedule rings exceed L2"},
        "roofline": {"bound": "alu", "achieved": ach, "peak": alu_peak, "unit": "Tops/s", "frac": ach / alu_peak,
                     "traffic": None, "kernel": "whole batched step (all kernels)"},
        "clocks": clk.summary(), "gpu_launches": pg.pamc_batch_launch_count(b) - l0,
    }
    emit(line)
    pg.pamc_batch_destroy(b)
    for h in hs:
        pg.pamc_destroy(h)


POTTS_PARAMS = dict(kind=1, R=2048, sweeps=10, steps=300, beta0=0.1, beta1=3.0, seed=0)
POTTS_WORKLOAD = "Max-3-Cut, random sparse N=2,000, m=12,000 (avg deg 12), unit weights, R=2048, 10 sweeps/step"


def run_potts(args):
    """Configuration 3: three-state Potts on the N=2,000 graph, the cascaded
    sampler (rule 0) as the headline and the softmax noisy argmax (rule 2,
    gamma 1) beside it; steps 0..K-1 of a fresh run timed with CUDA events."""
    import torch
    import paper_2606_25203_gb300 as pg
    pg.load()
    inst = W.c3_sparse2000()
    stream = torch.cuda.current_stream()
    flush = torch.empty(512 * 1024 * 1024 // 4, dtype=torch.int32, device="cuda")
    out = {}
    for name, extra in (("cascaded", dict(rule=0)), ("softmax", dict(rule=2, K=3, gamma=1.0))):
        P = dict(POTTS_PARAMS, **extra)
        s = pg.Solver(inst.row_ptr, inst.col, inst.w, stream=stream.cuda_stream)
        s.init(**P)
        s.step(args.warmup)
        s.sync()
        s.init(**P)
        torch.cuda.synchronize()
        l0 = s.launches()
        ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
              for _ in range(args.steps)]
        with ClockSampler(0) as clk:
            for k in range(args.steps):
                flush.add_(1)
                ev[k][0].record(stream)
                s.step(1)
                ev[k][1].record(stream)
            torch.cuda.synchronize()
        ms = sum(a.elapsed_time(b) for a, b in ev)
        cut, _ = s.best()
        out[name] = dict(ms=ms, launches=s.launches() - l0, cut=int(cut), clocks=clk.summary())
        s.close()
    att = POTTS_PARAMS["R"] * inst.n * POTTS_PARAMS["sweeps"] * args.steps
    deg = inst.nnz / inst.n
    peaks, _ = load_peaks()
    peak = 152 * 128 * peaks.get("sm_max_mhz", 2070.0) * 1e6 / 1e12
    # cascaded: half a Philox call (30 ops), 2 ops per incident edge, two threshold tests (8)
    ops = 30 + 2 * deg + 8
    c = out["cascaded"]
    ach = att * ops / (c["ms"] / 1e3) / 1e12
    line = {
        "metric": METRIC, "value": att / (c["ms"] / 1e3), "unit": "attempts/s", "n_gpus": 1,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": c["ms"] / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "int32",
        "data": "synthetic",
        "config": {"workload": POTTS_WORKLOAD, **POTTS_PARAMS, "l2": "flushed between steps (512 MB write)",
                   "timed_steps": f"steps 0..{args.steps - 1} of a fresh run"},
        "roofline": {"bound": "alu", "achieved": ach, "peak": peak, "unit": "Tops/s", "frac": ach / peak,
                     "traffic": None, "kernel": "whole step, k_sweep_potts (cascaded) dominating",
                     "ops_per_attempt": ops},
        "cut_after_timed_steps": c["cut"],
        "softmax": {"value": att / (out["softmax"]["ms"] / 1e3), "unit": "attempts/s",
                    "ms_per_step": out["softmax"]["ms"] / args.steps, "cut_after_timed_steps": out["softmax"]["cut"],
                    "gamma": 1.0},
        "clocks": c["clocks"], "gpu_launches": c["launches"],
    }
    emit(line)


# time-to-target runs: the paper's method (stagnation control and NCM on) on the Erdos-Renyi N=800 instance
TTS_PARAMS = dict(R=128, sweeps=5, steps=500, beta0=0.1, beta1=3.0, stagnation=1, z_rst=400, seed=0)


def run_tts(args):
    """Time-to-target cut (the paper's TTS: T_com ln(1-0.99) / ln(1-P_s)) on the
    Erdos-Renyi N=800 instance with the augmented controller (stagnation
    control and NCM on; R=128, 5 sweeps, 500 steps).  The target is the best cut
    of three long reference runs (R=1024, 1000 steps); then `args.tts_runs`
    independent runs stop when they reach it.  For every run length k, P_s(k)
    is the fraction of runs that reached the target within k steps and
    T_com(k) = k times the device time of a step; the reported TTS is the
    minimum over k (P_s = 1 counts as a single run)."""
    import math
    import torch
    import paper_2606_25203_gb300 as pg
    pg.load()
    inst = W.c1_er800()
    stream = torch.cuda.current_stream()
    target = -1
    for sd in range(3):
        s = pg.Solver(inst.row_ptr, inst.col, inst.w, stream=stream.cuda_stream)
        s.run(**dict(TTS_PARAMS, R=1024, steps=1000, seed=1000 + sd))
        target = max(target, int(s.best()[0]))
        s.close()
    # device time of one step of the configuration (no early stop)
    s = pg.Solver(inst.row_ptr, inst.col, inst.w, stream=stream.cuda_stream)
    s.init(**TTS_PARAMS)
    s.step(args.warmup)
    s.sync()
    s.init(**TTS_PARAMS)
    torch.cuda.synchronize()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with ClockSampler(0) as clk:
        a.record(stream)
        s.step(TTS_PARAMS["steps"])
        b.record(stream)
        torch.cuda.synchronize()
    ms_step = a.elapsed_time(b) / TTS_PARAMS["steps"]
    s.close()
    reach = []
    launches = 0
    t0 = time.perf_counter()
    for sd in range(args.tts_runs):
        s = pg.Solver(inst.row_ptr, inst.col, inst.w, stream=stream.cuda_stream)
        s.run(**dict(TTS_PARAMS, seed=sd, target_cut=target))
        c = s.control()
        reach.append(int(c["t"]) if c["done"] else None)
        launches += s.launches()
        s.close()
    wall = time.perf_counter() - t0
    best = None
    for k in range(1, TTS_PARAMS["steps"] + 1):
        ps = sum(1 for r in reach if r is not None and r <= k) / len(reach)
        if ps <= 0:
            continue
        t_com = k * ms_step / 1e3
        tts = t_com if ps >= 0.99 else t_com * math.log(0.01) / math.log(1.0 - ps)
        if best is None or tts < best[0]:
            best = (tts, k, ps, t_com)
    line = {
        "metric": "time-to-target cut (99%)", "value": best[0] if best else None, "unit": "s", "n_gpus": 1,
        "steps": TTS_PARAMS["steps"], "warmup": args.warmup, "ms_per_step": ms_step,
        "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": "int32", "data": "synthetic",
        "config": {"workload": "Erdos-Renyi N=800, p=0.06, unit weights; augmented PAMC, R=128, beta 0.1 -> 3.0 "
                               "over 500 steps, 5 sweeps/step, restart every 400", "runs": args.tts_runs,
                   "target": f"best cut of three reference runs (R=1024, 1000 steps): {target}"},
        "target_cut": target, "best_steps": best[1] if best else None, "P_s": best[2] if best else 0.0,
        "T_com_s": best[3] if best else None,
        "reached": sum(1 for r in reach if r is not None), "runs_wall_s": wall,
        "gpu_launches": launches, "clocks": clk.summary(),
    }
    emit(line)


def run_diag(args):
    """Diagnostics on the torus population of the default workload (R=4096):
    the corrected pairwise Hamming histogram (8.4M pairs) and the lineage,
    each timed as the whole C-ABI call (scratch, kernels, readback)."""
    import torch
    import paper_2606_25203_gb300 as pg
    pg.load()
    inst = W.c2a_torus141()
    h = pg.pamc_create_csr(inst.n, inst.row_ptr, inst.col, inst.w)
    pg.pamc_init(h, **PARAMS)
    pg.pamc_step(h, 5)
    pg.pamc_sync(h)
    for _ in range(args.warmup):
        pg.pamc_hamming(h, inst.n)
    ts = []
    with ClockSampler(0) as clk:
        for _ in range(args.steps):
            t0 = time.perf_counter()
            hist, total = pg.pamc_hamming(h, inst.n)
            ts.append(time.perf_counter() - t0)
    t1 = time.perf_counter()
    fam, nf = pg.pamc_lineage(h, R)
    t_lin = time.perf_counter() - t1
    pairs = R * (R - 1) // 2
    nw = (inst.n + 31) // 32
    sec = float(np.median(ts))
    peaks, peak_src = load_peaks()
    if os.environ.get("PAMC_HAMMING") == "cuda":
        ops = pairs * nw * 3                    # xor, popcount, add per word pair
        peak = 152 * 128 * peaks.get("sm_max_mhz", 2070.0) * 1e6 / 1e12
        roof = {"bound": "alu", "achieved": ops / sec / 1e12, "peak": peak, "unit": "Tops/s",
                "frac": ops / sec / 1e12 / peak, "traffic": None, "kernel": "k_hamming (XOR-popcount)"}
    else:
        # the overlaps of every pair i < j: 2 n flops each, on fp8 tensor cores
        # (peak: the measured bf16 burst x 2, the nominal fp8 / bf16 ratio)
        flops = pairs * 2 * inst.n
        peak = 2 * peaks.get("bf16_tflops", 1900.0)
        roof = {"bound": "tensor", "achieved": flops / sec / 1e12, "peak": peak, "unit": "TFLOP/s",
                "frac": flops / sec / 1e12 / peak, "traffic": None,
                "kernel": "k_hamming_tc (tcgen05 kind::f8f6f4, whole call timed)",
                "peak_source": f"{peak_src} bf16 burst x 2"}
    line = {
        "metric": "replica pairs/s (Hamming histogram)", "value": pairs / sec, "unit": "pairs/s", "n_gpus": 1,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": sec * 1e3, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "u32", "data": "synthetic",
        "config": {"workload": "torus 141x141, R=4096 after 5 steps of the default run", "pairs": pairs,
                   "timing": "median host wall clock of the whole pamc_hamming call"},
        "roofline": roof,
        "mean_normalised_distance": total / (pairs * inst.n), "lineage_ms": t_lin * 1e3,
        "families_alive": nf, "clocks": clk.summary(), "gpu_launches": 2 * args.steps,
    }
    emit(line)
    pg.pamc_destroy(h)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=None,
                    help="timed steps (default: the whole 500-step schedule for the sparse workload, 20 otherwise)")
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--only", choices=["torus", "sparse"], default=None,
                    help="run one of the two instances (profiling)")
    ap.add_argument("--lean", action="store_true",
                    help="timed steps only: no e2e, kernel split or CPU baseline (profiling)")
    ap.add_argument("--workload", choices=["sparse", "dense100k", "serving", "batch", "diag", "potts", "tts"],
                    default="sparse")
    ap.add_argument("--batch-requests", type=int, default=48)
    ap.add_argument("--tts-runs", type=int, default=32)
    ap.add_argument("--batch-n-lo", type=int, default=800)
    ap.add_argument("--batch-n-hi", type=int, default=20000)
    ap.add_argument("--serve-requests", type=int, default=48)
    ap.add_argument("--serve-max3cut", type=float, default=0.25,
                    help="fraction of the serving requests that ask for Max-3-Cut")
    ap.add_argument("--serve-max-active", type=int, default=64)
    ap.add_argument("--dense-n", type=int, default=DENSE_N)
    ap.add_argument("--dense-e2e", action="store_true", help="dense100k: add the end-to-end figure")
    ap.add_argument("--one-stream", action="store_true",
                    help="sparse workload: step the two instances one after the other on one stream")
    ap.add_argument("--no-dense", action="store_true",
                    help="sparse workload: leave out the dense100k object (profiling)")
    ap.add_argument("--replicas", action="store_true",
                    help="several GPUs: independent populations (own seed each) instead of one split population")
    ap.add_argument("--split", action="store_true",
                    help="one GPU: run the split-population path (the exchange over a group of one)")
    args = ap.parse_args()
    if args.steps is None:
        args.steps = STEPS_SCHEDULE if (args.workload == "sparse" and args.impl == "ours") else 20
    global ONLY
    ONLY = args.only
    if args.workload == "dense100k" and args.impl == "ours":
        run_dense(args)
        return
    if args.workload == "tts" and args.impl == "ours":
        run_tts(args)
        return
    if args.workload == "potts" and args.impl == "ours":
        run_potts(args)
        return
    if args.workload == "diag" and args.impl == "ours":
        run_diag(args)
        return
    if args.workload == "batch" and args.impl == "ours":
        run_batch(args)
        return
    if args.workload == "serving" and args.impl == "ours":
        run_serving(args)
        return
    if args.impl == "reference":
        rank = int(os.environ.get("RANK", "0"))
        if rank != 0:
            return
        run_reference(args)
        return
    run_ours(args)


if __name__ == "__main__":
    sys.stdout.flush()
    JSON_OUT = os.fdopen(os.dup(1), "w")
    os.dup2(2, 1)
    main()
