"""Benchmark: greedy multi-hit WSC solves per second on one or more GB300s.

A step is one whole greedy solve (every round of Algorithm 1 with its P-DFS
argmax, §III-D) of the synthetic cohort "c2" (h=3, G=5,000, Nt=500, Nn=300,
seed 1; see synth/), with the cohort already resident on the device.  Between
timed steps a 256 MiB buffer is written to flush L2 (the cohort is far smaller
than L2).  Each step is timed with CUDA events on the solving stream; the timed
region is bracketed by barrier + synchronize; the result is the max over ranks.
On one GPU the line also carries the batched workload (16 uneven cohorts in one
launch against one after another) and the served one (a request trace replayed
against the continuous-batching server and against a plain loop).

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

N > 1 runs under torchrun: every rank solves its own copy of the workload (weak
scaling, no collective on the data path).  --impl reference times the CPU P-DFS
of oracle/ (threaded over every host core, checked against the single-threaded
oracle) solving the same workload, one whole solve per step.

The line's roofline compares the solve kernel's executed integer work (from the
committed ncu capture of the same kernel source) with this GPU's measured LOP3
rate; cpu_baseline is measured on this host without extrapolation; plain_configs
adds the c1 and c3 single-cohort solves.
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
sys.path.insert(0, ROOT)

METRIC = "wsc_solves_per_s"
UNIT = "solves/s"
WORKLOAD = "c2"
H, ALPHA = 3, (1, 10)


def _dist_env():
    return int(os.environ.get("RANK", 0)), int(os.environ.get("WORLD_SIZE", 1)), int(os.environ.get("LOCAL_RANK", 0))


def aggregate_max(values, world):
    """Max over ranks of each value (identity on one rank)."""
    if world == 1:
        return list(values)
    import torch
    import torch.distributed as dist
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor(list(values), dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return t.cpu().tolist()


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


class ClockSampler:
    """nvidia-smi samples of SM clock and throttle reasons during the timed region."""
    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.QUERY}",
                                          "--format=csv,noheader,nounits", "-lms", "50"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
            # the timed region starts once nvidia-smi is sampling (at most 3 s)
            t0 = time.time()
            while not self.lines and time.time() - t0 < 3.0 and self.proc.poll() is None:
                time.sleep(0.01)
            self.lines.clear()
        except (OSError, FileNotFoundError):
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
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.thread.join(timeout=2)
        sm, smax, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                smax = float(f[2])
            except ValueError:
                continue
            for name, v in zip(names, f[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(name)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": smax,
                "reasons": sorted(reasons), "samples": len(sm)}


def algorithmic_ops(r, Nt, Nn):
    """32-bit integer operations the P-DFS of §III-D performs for a solve's counters.

    Per unit, with w_t = 2 * ceil(Nt / 64) and w_n = 2 * ceil(Nn / 64) 32-bit words
    per tumor / normal row: every visited node at every depth costs w_t LOP3 (the
    AND with the parent's intersection fused with the zero test) + 1 compare; every
    scored leaf (TP > 0) additionally w_t AND + w_t POPC + w_n AND + w_n POPC + 6
    (score, key and compare).  Returns (ops of the whole solve, ops of the leaves)."""
    wt = 2 * ((Nt + 63) // 64)
    wn = 2 * ((Nn + 63) // 64)
    visited_all = int(r.visited.sum())
    visited_leaf = int(r.visited[:, -1].sum())
    scored = int((r.visited[:, -1] - r.pruned[:, -1]).sum())
    per_scored = 2 * wt + 2 * wn + 6
    return visited_all * (wt + 1) + scored * per_scored, visited_leaf * (wt + 1) + scored * per_scored


def kernel_source_sha256():
    """Of the files that the solve kernel is made of, one after another."""
    import hashlib
    sha = hashlib.sha256()
    for name in ("mh_kernels.cu", "mh_levels.cuh", "mh_barrier.h", "mh_internal.h"):
        with open(os.path.join(ROOT, "paper_2603_16721_gb300", "csrc", name), "rb") as f:
            sha.update(f.read())
    return sha.hexdigest()


def _profiled_fields(kernel_file="k_solve_c2.md"):
    """Fields of the committed ncu summary of the solve kernel ("- `key`: `value`"
    lines), if that summary was taken from the kernel source as it is now (else {})."""
    try:
        text = open(os.path.join(ROOT, "profiles", kernel_file)).read()
        sha = kernel_source_sha256()
    except OSError:
        return {}
    fields = {k: v.strip("`") for k, v in (ln.strip("- `").split(": ", 1) for ln in text.splitlines()
                                             if ln.startswith("- `") and ": " in ln)}
    return fields if fields.get("kernel_source_sha256") == sha else {}


def _profiled_int(key, kernel_file="k_solve_c2.md"):
    try:
        return int(float(_profiled_fields(kernel_file)[key]))
    except (KeyError, ValueError):
        return None


def int_peaks():
    """Measured integer throughput of this GPU (thread ops/s): LOP3 and POPC."""
    from paper_2603_16721_gb300 import mh
    lop3, _ = mh.mh_int_peak(0)
    popc, _ = mh.mh_int_peak(1)
    return {"lop3_tops": lop3 / 1e12, "popc_tops": popc / 1e12}


def solve_roofline(res_list, Nt, Nn, peaks_int, kernel_file="k_solve_c2.md"):
    """Integer-pipe roofline of the persistent solve kernel (the dominant kernel:
    one cooperative launch runs every round of a solve).

    achieved = the integer and logic thread instructions one launch executes
    (sm__sass_thread_inst_executed_op_integer_pred_on + ..._op_bit_pred_on, from
    the committed ncu capture of this kernel source on the same workload) / the
    launch's duration measured here (CUDA events around each cooperative launch on
    the solving stream); peak = the measured LOP3 rate of this GPU (mh_int_peak).
    work_equiv = the paper's per-node cost of the same search (algorithmic_ops,
    units: every visited node and scored leaf of the exact counters, each at the
    per-node cost of a node-by-node search)
    over the same duration: the rate a kernel doing the paper's work would need;
    the kernel reaches the same counters with far fewer operations, so this is not
    pipe utilisation."""
    ops = [algorithmic_ops(r, Nt, Nn) for r in res_list]
    kernel_s = sum(r.kernel_ms for r in res_list) / 1e3
    launches = sum(max(1, r.kernel_launches - 1) for r in res_list)  # minus the init kernel
    if kernel_s <= 0:
        return None
    avg_s = kernel_s / launches
    peak = peaks_int["lop3_tops"]
    executed = _profiled_int("int_thread_ops_per_launch", kernel_file)
    achieved = executed / avg_s / 1e12 if executed else None
    wequiv = sum(o[0] for o in ops) / launches / avg_s / 1e12
    prof = _profiled_fields(kernel_file)
    ncu = {k: float(prof[k]) for k in ("alu_pipe_active_pct", "issue_active_pct", "warps_active_pct",
                                       "barrier_stall_per_issue", "duration_ms") if k in prof} or None
    return {"bound": "alu", "achieved": round(achieved, 4) if achieved else None, "peak": round(peak, 3),
            "unit": "Tops/s (int32 thread ops)", "frac": round(achieved / peak, 4) if achieved else None,
            "traffic": _profiled_int("dram_bytes_per_launch", kernel_file),
            "kernel": "k_solve (persistent solve, one launch per solve)", "launches": launches,
            "avg_launch_us": round(avg_s * 1e6, 2), "executed_int_ops_per_launch": executed,
            "peak_source": "measured: mh_int_peak LOP3 rate on this GPU (popc rate in int_peaks)",
            "int_peaks": {k: round(v, 3) for k, v in peaks_int.items()},
            "work_equiv": {"ops_per_launch": round(sum(o[0] for o in ops) / launches),
                           "achieved": round(wequiv, 4), "work_equiv_frac": round(wequiv / peak, 4)},
            "ncu": ncu,
            "latency": latency_chain(res_list, avg_s)}


def latency_chain(res_list, avg_s):
    """The solve's time in the unit that bounds it: a round is a chain of dependent
    steps (block barriers, the grid barrier, L2 round trips), so the kernel's time
    per round is given beside one dependent L2 load measured on this GPU
    (mh_l2_latency), as the number of such loads it equals."""
    from paper_2603_16721_gb300 import mh
    try:
        ns = mh.mh_l2_latency()
    except Exception:  # a diagnostic: the line stands without it
        return None
    rounds = sum(r.rounds for r in res_list) / max(1, len(res_list))
    us_round = avg_s * 1e6 / max(1.0, rounds)
    return {"rounds_per_launch": rounds, "us_per_round": round(us_round, 3),
            "l2_dependent_load_us": round(ns / 1e3, 4),
            "l2_loads_per_round": round(us_round * 1e3 / ns, 1) if ns > 0 else None}


def cpu_threads():
    import oracle
    return oracle.default_threads()


def cpu_baseline_measure(c):
    """CPU baselines on this host, measured (no extrapolation): the threaded CPU
    P-DFS (oracle/pdfs_mt.c, every host core, the paper's master-worker scheme on
    threads) solving the whole workload once; the single-threaded oracle P-DFS on
    its first two greedy rounds; the brute-force oracle on the whole c1 solve."""
    import oracle
    import synth
    th = cpu_threads()
    t0 = time.perf_counter()
    sol = oracle.pdfs_mt(c.bitmaps, c.G, c.Nt, c.Nn, H, ALPHA, threads=th)
    dt = time.perf_counter() - t0
    t0 = time.perf_counter()
    one = oracle.pdfs(c.bitmaps, c.G, c.Nt, c.Nn, H, ALPHA, max_rounds=2)
    dt1 = time.perf_counter() - t0
    c1 = synth.generate(synth.c1())
    t0 = time.perf_counter()
    bf = oracle.bruteforce(c1.bitmaps, c1.G, c1.Nt, c1.Nn, 2, ALPHA)
    dtb = time.perf_counter() - t0
    return {"value": 1.0 / dt, "unit": UNIT, "cores": th, "kind": "oracle",
            "sample": f"threaded CPU P-DFS (oracle/pdfs_mt.c, {th} threads) solving the whole {WORKLOAD} workload "
                      f"once ({sol.k} selections, {sol.visited.shape[0]} rounds): {dt:.2f} s",
            "single_thread_oracle": {"rounds": int(one.visited.shape[0]), "seconds": round(dt1, 3),
                                     "visited_nodes": int(one.visited.sum()), "cores": 1,
                                     "what": f"oracle P-DFS (plain C), first 2 greedy rounds of {WORKLOAD}"},
            "bruteforce_c1": {"seconds": round(dtb, 3), "selections": bf.k, "cores": 1,
                              "what": "brute-force oracle (every 2-subset, no pruning), whole c1 solve"}}


def run_reference(args):
    """Reference arm: the CPU P-DFS of oracle/ (threaded over every host core) solving
    the whole c2 workload once per step; ms_per_step is what each step took."""
    rank, world, _ = _dist_env()
    if world > 1 and rank != 0:
        return 0
    import oracle
    import synth
    c = synth.generate(synth.c2())
    th = cpu_threads()
    times = []
    k = rounds = 0
    for i in range(args.warmup + args.steps):
        t0 = time.perf_counter()
        sol = oracle.pdfs_mt(c.bitmaps, c.G, c.Nt, c.Nn, H, ALPHA, threads=th)
        dt = time.perf_counter() - t0
        k, rounds = sol.k, int(sol.visited.shape[0])
        if i >= args.warmup:
            times.append(dt)
    total = sum(times)
    value = len(times) / total
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * total / len(times),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u64", "data": "synthetic",
            "config": {"workload": "c2: h=3, G=5000, Nt=500, Nn=300, seed 1, alpha=1/10"},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": th, "kind": "oracle",
                             "sample": f"threaded CPU P-DFS (oracle/pdfs_mt.c, {th} threads), one whole c2 solve "
                                       f"per step ({k} selections, {rounds} rounds)"},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line))
    return 0


def run_ours(args):
    import torch
    rank, world, local = _dist_env()
    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    torch.cuda.set_device(local)
    import __graft_entry__
    __graft_entry__.build()
    import synth
    from paper_2603_16721_gb300 import mh

    c = synth.generate(synth.c2())
    stream = torch.cuda.Stream()
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    H = mh.mh_create(c.bitmaps, c.G, c.Nt, c.Nn)
    mh.mh_set_stream(H, stream.cuda_stream)
    for _ in range(args.warmup):
        mh.mh_solve_ex(H, H_HITS, ALPHA, max_rounds=args.max_rounds, mode=MODES[args.mode])
    torch.cuda.synchronize()

    sampler = ClockSampler(torch.cuda.current_device()) if rank == 0 else None
    results, step_ms = [], []
    barrier(world)
    torch.cuda.synchronize()
    if sampler:
        sampler.start()
    for _ in range(args.steps):
        with torch.cuda.stream(stream):
            flush.fill_(1)
        ev0 = torch.cuda.Event(enable_timing=True)
        ev1 = torch.cuda.Event(enable_timing=True)
        ev0.record(stream)
        r = mh.mh_solve_ex(H, H_HITS, ALPHA, max_rounds=args.max_rounds, time_kernels=True, mode=MODES[args.mode])
        ev1.record(stream)
        ev1.synchronize()
        step_ms.append(ev0.elapsed_time(ev1))
        results.append(r)
    torch.cuda.synchronize()
    barrier(world)
    clocks = sampler.stop() if sampler else None
    total_ms = sum(step_ms)
    total_ms_max, = aggregate_max([total_ms], world)
    value = world * args.steps / (total_ms_max / 1e3)

    if args.kernels_only:  # profiling run: the timed solves only
        H.close()
        if rank == 0:
            print(json.dumps({"kernels_only": True, "ms_per_step": total_ms / args.steps}))
        return 0

    # end to end through the C ABI with host buffers: create (H2D), solve, read back
    e2e_ms = []
    d2h = 0
    for _ in range(max(2, min(args.steps, 5))):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        with mh.mh_create(c.bitmaps, c.G, c.Nt, c.Nn) as H2:
            r2 = mh.mh_solve(H2, H_HITS, ALPHA)
        e2e_ms.append((time.perf_counter() - t0) * 1e3)
        d2h = r2.genes.nbytes + r2.tp.nbytes + r2.fp.nbytes + r2.visited.nbytes + r2.pruned.nbytes
    e2e_max, = aggregate_max([statistics.median(e2e_ms)], world)
    H.close()

    if rank == 0:
        r0 = results[-1]
        scored = int((r0.visited[:, -1] - r0.pruned[:, -1]).sum())
        vis_leaves = int(r0.visited[:, -1].sum())
        pruned_prefixes = int(r0.pruned[:, :-1].sum())
        cb = cpu_baseline_measure(c) if world == 1 else None
        peaks = int_peaks()
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": total_ms_max / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "u64", "data": "synthetic",
            "config": {"workload": "c2: h=3, G=5000, Nt=500, Nn=300, seed 1, alpha=1/10",
                       "parallelism": f"replicas x{world}", "l2": "flushed between steps (256 MiB write)",
                       "rounds_per_solve": r0.rounds, "selected": r0.k},
            "breakdown_ms_per_solve": {k: round(sum(getattr(r, k) for r in results) / len(results), 3)
                                       for k in ("level1_ms", "expand_ms", "leaf_ms", "finalize_ms")},
            "mode": "persistent" if r0.mode == mh.MH_MODE_PERSISTENT else "launches",
            "warp_balance": {k: {"mean_warp_cycles": round(r0.diag[i] / max(1, r0.diag[4 + i]), 1),
                                 "longest_warp_cycles_per_round": round(r0.diag[2 + i] / max(1, r0.rounds), 1)}
                             for i, k in enumerate(("expand", "leaf"))},
            "extra": {"p50_ms": statistics.median(step_ms), "p99_ms": sorted(step_ms)[int(0.99 * (len(step_ms) - 1))],
                      "combos_scored_per_s": scored * value / world, "leaves_tested_per_s": vis_leaves * value / world,
                      "prefixes_pruned_per_s": pruned_prefixes * value / world,
                      "visited_fraction": vis_leaves / (r0.rounds * _comb(c.G, H_HITS))},
            "roofline": solve_roofline(results, c.Nt, c.Nn, peaks),
            "cpu_baseline": cb,
            "e2e": {"value": world / (e2e_max / 1e3), "unit": UNIT,
                    "h2d_bytes_per_step": int(c.bitmaps.nbytes), "d2h_bytes_per_step": int(d2h)},
            "gpu_launches": int(sum(r.kernel_launches for r in results)),
            "clocks": clocks,
        }
        if world == 1 and not args.no_extras:
            # the other plain single-cohort configurations (c1: h=2, G=1,000; c3: h=4,
            # G=19,000, 128-bit rows): CUDA events on the solving stream, L2 flushed
            line["plain_configs"] = {"c1": plain_config("c1", 5, peaks), "c3": plain_config("c3", 3, peaks)}
            line["bound_mode"] = bound_comparison(c)
            line["train_test"] = train_test_coverage()
            # the other two parts of the metric, after the timed c2 steps: batched
            # (16 uneven cohorts in one launch vs one after another) and served
            # (request trace: continuous batching vs a plain loop)
            b16 = batch16_comparison(argparse.Namespace(steps=3, warmup=1))
            line["batched"] = {k: b16[k] for k in ("value", "unit", "sequential_value", "speedup_vs_sequential",
                                                   "identical_to_sequential", "config")}
            line["served"] = served_comparison(argparse.Namespace(requests=200, slots=8, large_slots=0))
        print(json.dumps(line))
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()
    return 0


def plain_config(name, runs, peaks_int=None):
    """One plain single-cohort configuration: the median of `runs` solves (after one
    warm-up) of its synthetic cohort, timed with CUDA events, L2 flushed between;
    with the measured integer peaks, the solve kernel's roofline when a committed ncu
    summary of the current kernel source on this configuration exists."""
    import torch
    import synth
    from paper_2603_16721_gb300 import mh
    spec = synth.COHORTS[name]()
    c = synth.generate(spec)
    stream = torch.cuda.Stream()
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    ms, kms, rs = [], [], []
    with mh.mh_create(c.bitmaps, c.G, c.Nt, c.Nn) as Hc:
        mh.mh_set_stream(Hc, stream.cuda_stream)
        r = mh.mh_solve(Hc, spec.h, ALPHA)
        for _ in range(runs):
            with torch.cuda.stream(stream):
                flush.fill_(1)
            ev0 = torch.cuda.Event(enable_timing=True)
            ev1 = torch.cuda.Event(enable_timing=True)
            ev0.record(stream)
            r = mh.mh_solve(Hc, spec.h, ALPHA)
            ev1.record(stream)
            ev1.synchronize()
            ms.append(ev0.elapsed_time(ev1))
            kms.append(r.kernel_ms)
            rs.append(r)
    t = statistics.median(ms) / 1e3
    scored = int((r.visited[:, -1] - r.pruned[:, -1]).sum())
    return {"workload": f"{name}: h={spec.h}, G={c.G}, Nt={c.Nt}, Nn={c.Nn}, seed {spec.seed}, alpha=1/10",
            "ms_per_solve": round(1e3 * t, 3), "kernel_ms_per_solve": round(statistics.median(kms), 3),
            "solves_per_s": round(1.0 / t, 3), "rounds": r.rounds, "selected": r.k,
            "combos_scored_per_s": scored / t, "leaves_tested_per_s": int(r.visited[:, -1].sum()) / t,
            "prefixes_pruned_per_s": int(r.pruned[:, :-1].sum()) / t,
            "visited_fraction": int(r.visited[:, -1].sum()) / (r.rounds * _comb(c.G, spec.h)), "runs": runs,
            "roofline": (solve_roofline(rs, c.Nt, c.Nn, peaks_int, f"k_solve_{name}.md")
                         if peaks_int and _profiled_fields(f"k_solve_{name}.md") else None)}


def bound_comparison(c):
    """The score-bound mode on the timed workload: same selections, fewer nodes."""
    import torch
    from paper_2603_16721_gb300 import mh
    out = {}
    rounds = 1
    with mh.mh_create(c.bitmaps, c.G, c.Nt, c.Nn) as Hb:
        for name, prune in (("paper", mh.MH_PRUNE_PAPER), ("bound", mh.MH_PRUNE_BOUND)):
            r = mh.mh_solve_ex(Hb, H_HITS, ALPHA, prune=prune)
            ms = []
            for _ in range(3):
                torch.cuda.synchronize()
                r = mh.mh_solve_ex(Hb, H_HITS, ALPHA, prune=prune)
                ms.append(r.kernel_ms)
            rounds = r.rounds
            out[name] = {"kernel_ms_per_solve": round(statistics.median(ms), 3), "records": r.records(),
                         "visited_leaves": int(r.visited[:, -1].sum()), "visited_nodes": int(r.visited.sum()),
                         "cut_prefixes": int(r.cut.sum())}
    same = out["paper"].pop("records") == out["bound"].pop("records")
    full = rounds * _comb(c.G, H_HITS)
    return {"identical_selections": same,
            "visited_fraction_paper": out["paper"]["visited_leaves"] / full,
            "visited_fraction_bound": out["bound"]["visited_leaves"] / full,
            "paper": out["paper"], "bound": out["bound"],
            "note": "bound mode runs the node-by-node search (no per-sample sums); its counters depend on "
                    "when candidates were found"}


def train_test_coverage():
    """§IV-D on the synthetic workload: learn on 75% of c2's samples, evaluate the
    frozen combinations on the training and held-out samples (GPU coverage)."""
    import synth
    from paper_2603_16721_gb300 import mh
    c = synth.generate(synth.c2())
    (tr, nt, nn), (te, mt, mn) = synth.split_samples(c, 0.75, seed=7)
    with mh.mh_create(tr, c.G, nt, nn) as Ht:
        sol = mh.mh_solve(Ht, H_HITS, ALPHA)
        train = mh.mh_evaluate(Ht, sol.genes)
    with mh.mh_create(te, c.G, mt, mn) as He:
        test = mh.mh_evaluate(He, sol.genes)
    keys = ("tc", "tt", "nc", "nt", "sensitivity", "specificity")
    return {"workload": "c2 samples split 75/25 (seed 7): learn on train, evaluate on both",
            "combinations": sol.k, "train": {k: train[k] for k in keys}, "test": {k: test[k] for k in keys}}


def _comb(n, k):
    import math
    return math.comb(n, k)


H_HITS = H
MODES = {"persistent": 0, "launches": 1}


def run_batch16(args):
    print(json.dumps(batch16_comparison(args)))
    return 0


def batch16_comparison(args):
    """Batched workload: 16 cohorts of uneven size (seeds 100-115, h=3 for 12, h=4 for 4)
    solved in one persistent launch, against the same 16 solved one after another."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import synth
    from paper_2603_16721_gb300 import mh
    specs = synth.batch16()
    cohorts = [synth.generate(sp) for sp in specs]
    stream = torch.cuda.Stream()
    handles = [mh.mh_create(c.bitmaps, c.G, c.Nt, c.Nn) for c in cohorts]
    for H in handles:
        mh.mh_set_stream(H, stream.cuda_stream)
    hs = [sp.h for sp in specs]
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    # sequential plain solves (one persistent launch per solve)
    seq = []
    for _ in range(args.warmup + args.steps):
        with torch.cuda.stream(stream):
            flush.fill_(1)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        rs = [mh.mh_solve(H, h) for H, h in zip(handles, hs)]
        seq.append(time.perf_counter() - t0)
    seq_t = statistics.median(seq[args.warmup:])
    # batched solves (the first call autotunes the block split)
    bat = []
    for _ in range(args.warmup + args.steps):
        with torch.cuda.stream(stream):
            flush.fill_(1)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        rb = mh.mh_solve_batch(handles, hs)
        bat.append(time.perf_counter() - t0)
    bat_t = statistics.median(bat[args.warmup:])
    same = all(a.records() == b.records() for a, b in zip(rs, rb))
    out = ({
        "metric": "batched_wsc_solves_per_s", "value": len(handles) / bat_t, "unit": "solves/s",
        "sequential_value": len(handles) / seq_t, "speedup_vs_sequential": seq_t / bat_t,
        "identical_to_sequential": same, "steps": args.steps, "warmup": args.warmup,
        "config": {"workload": "batch16: 16 cohorts, seeds 100-115, G~U[2000,19000], Nt~U[100,1000], "
                               "Nn~U[50,500], h=3 x12 and h=4 x4, alpha=1/10"},
        "per_cohort": [{"G": c.G, "Nt": c.Nt, "Nn": c.Nn, "h": sp.h, "k": r.k, "rounds": r.rounds,
                        "solo_ms": round(r.solve_ms, 3)} for c, sp, r in zip(cohorts, specs, rs)],
    })
    for H in handles:
        H.close()
    return out


def run_served(args):
    print(json.dumps(served_comparison(args)))
    return 0


def served_comparison(args):
    """Served workload: a trace of requests (c3-law cohorts, Poisson arrivals at 5/s,
    h from {2: .3, 3: .5, 4: .2}) replayed in real time against (i) the served
    runtime (continuous batching) and (ii) a plain FIFO loop of one solve (one
    persistent launch) per request; latency = arrival to result.  The same trace is
    replayed again with its arrival times compressed so that the offered load is
    0.8x the plain loop's measured capacity, and finally every request arrives at
    once (saturated): each of the three is run on both paths."""
    import threading
    import numpy as np
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import synth
    from paper_2603_16721_gb300 import mh
    specs, gaps = synth.served200()
    n = min(args.requests, len(specs))
    specs = specs[:n]
    arrivals = np.cumsum(gaps[:n]) - gaps[0]
    cohorts = [synth.generate(sp) for sp in specs]
    torch.cuda.synchronize()
    # warm-up: one request of each h, both paths
    for h in (2, 3, 4):
        c = next(c for c, sp in zip(cohorts, specs) if sp.h == h)
        with mh.mh_create(c.bitmaps, c.G, c.Nt, c.Nn) as H:
            mh.mh_solve(H, h)

    def pct(xs, q):
        xs = sorted(xs)
        return xs[min(len(xs) - 1, int(round(q * (len(xs) - 1))))]

    def plain(arr):
        """Plain FIFO loop: returns results, latencies, service times, span."""
        res, lat, service = [], [], []
        t0 = time.perf_counter()
        for i, (c, sp) in enumerate(zip(cohorts, specs)):
            now = time.perf_counter() - t0
            if now < arr[i]:
                time.sleep(arr[i] - now)
            ts = time.perf_counter()
            with mh.mh_create(c.bitmaps, c.G, c.Nt, c.Nn) as H:
                res.append(mh.mh_solve(H, sp.h))
            te = time.perf_counter()
            service.append(te - ts)
            lat.append(te - t0 - arr[i])
        return res, lat, service, time.perf_counter() - t0

    def served(S, arr):
        """Requests submitted at their arrival times; returns results, latencies, span."""
        tickets = [None] * n
        t0 = time.perf_counter()

        def submitter():
            for i, (c, sp) in enumerate(zip(cohorts, specs)):
                now = time.perf_counter() - t0
                if now < arr[i]:
                    time.sleep(arr[i] - now)
                tickets[i] = S.submit(c.bitmaps, c.G, c.Nt, c.Nn, sp.h)

        th = threading.Thread(target=submitter)
        th.start()
        th.join()
        res = [S.wait(t) for t in tickets]
        return res, [r.solve_ms / 1e3 for r in res], time.perf_counter() - t0

    def summary(lat, span):
        return {"solves_per_s": n / span, "p50_ms": 1e3 * pct(lat, 0.50), "p99_ms": 1e3 * pct(lat, 0.99)}

    plain_res, plain_lat, service, plain_span = plain(arrivals)
    mean_service = sum(service) / n
    capacity = 1.0 / mean_service
    scale = (n / max(arrivals[-1], 1e-9)) / (0.8 * capacity)  # 5 req/s -> 0.8x capacity
    fast = arrivals * scale
    zero = np.zeros(n)
    pl_fast_res, pl_fast_lat, _, pl_fast_span = plain(fast)
    pl_burst_res, pl_burst_lat, _, pl_burst_span = plain(zero)
    with mh.Server(slots=args.slots, large_slots=args.large_slots) as S:
        served_res, served_lat, served_span = served(S, arrivals)
        fast_res, fast_lat, fast_span = served(S, fast)
        burst_res, burst_lat, burst_span = served(S, zero)
        stats = S.stats()
    same = all(a.records() == b.records() for a, b in zip(plain_res, served_res))
    for other in (fast_res, burst_res, pl_fast_res, pl_burst_res):
        same = same and all(a.records() == b.records() for a, b in zip(plain_res, other))
    return ({
        "metric": "served_wsc_solves_per_s", "value": n / served_span, "unit": "solves/s",
        "p50_ms": 1e3 * pct(served_lat, 0.50), "p99_ms": 1e3 * pct(served_lat, 0.99),
        "plain": {"value": n / plain_span, "p50_ms": 1e3 * pct(plain_lat, 0.50), "p99_ms": 1e3 * pct(plain_lat, 0.99),
                  "mean_service_ms": 1e3 * mean_service, "capacity_solves_per_s": capacity},
        "load_0p8": {"offered_req_per_s": n / max(fast[-1], 1e-9), "served": summary(fast_lat, fast_span),
                     "plain": summary(pl_fast_lat, pl_fast_span)},
        "saturated": {"served": summary(burst_lat, burst_span), "plain": summary(pl_burst_lat, pl_burst_span)},
        "offered_load_req_per_s": n / max(arrivals[-1], 1e-9), "requests": n, "slots": args.slots,
        "identical_to_plain": same, "server_launches": stats["launches"],
        "config": {"workload": f"served: first {n} of 200 requests, c3-law cohorts (G=19000, Nt=800, Nn=400), "
                               "seeds 1000-1199, Poisson 5 req/s, h from {2:.3,3:.5,4:.2}, trace seed 5000; "
                               "replayed as traced, compressed to 0.8x the plain loop's capacity, and all at once"},
    })


def main(argv=None):
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--max-rounds", type=int, default=0, help="stop each solve after R rounds (profiling)")
    ap.add_argument("--kernels-only", action="store_true", help="time the solves only (profiling runs)")
    ap.add_argument("--no-extras", action="store_true",
                    help="c2: leave out the batched and served comparisons appended to the line")
    ap.add_argument("--mode", choices=["persistent", "launches"], default="persistent",
                    help="one persistent kernel per solve, or one launch per phase")
    ap.add_argument("--workload", choices=["c2", "c1", "c3", "batch16", "served200"], default="c2",
                    help="c2: the headline single-cohort solve; c1, c3: the other plain solves (their timing "
                         "alone, --steps runs); batch16: the batched workload; served200: the served request trace")
    ap.add_argument("--requests", type=int, default=200, help="served200: requests replayed")
    ap.add_argument("--slots", type=int, default=8, help="served200: concurrent requests")
    ap.add_argument("--large-slots", type=int, default=0,
                    help="served200: large requests solved concurrently (0: the library default)")
    args = ap.parse_args(argv)
    if args.impl == "reference":
        return run_reference(args)
    if args.workload == "batch16":
        return run_batch16(args)
    if args.workload == "served200":
        return run_served(args)
    if args.workload in ("c1", "c3"):
        import __graft_entry__
        __graft_entry__.build()
        print(json.dumps(plain_config(args.workload, max(1, args.steps))))
        return 0
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
