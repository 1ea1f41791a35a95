#!/usr/bin/env python3
"""Throughput benchmark of the SneakySnake filter on GB300; prints one JSON
line.

Workload (short-read threshold sweep): 30,000,000 read/reference pairs of
100 bp, seeded and synthetic -- even pairs carry Poisson(3) random edits,
odd pairs are independent random sequences (the shape of the paper's
100 bp datasets, Section 3.1) -- filtered at E = 0, 2, 4, 6, 8, 10.

One step = the whole hot path over the batch: pack the resident ASCII reads
and references to 2 bits per base in the bit-sliced layout (SS_FMT_SLICED2,
2 launches) and filter it at every threshold with one ss_filter_sweep
call, 32 pairs per thread: E = 0, 2 and 4 in one shared pass over the pairs
(their walks cost less than reading the pairs), E = 6, 8 and 10 one launch
each (4 launches, side by side on the library's streams so that the GPU
does not drain between them).  ``value`` counts pair decisions (pairs x
thresholds) per second with the inputs resident in HBM; the inputs (6 GB
ASCII + 1.5 GB packed) are far larger than L2, so no flush is needed.
``pair_major_form`` times the same step with the pair-major packed format
and its one-pair-per-thread kernel, beside the headline.
``e2e`` runs the same sweep through ``ss_filter_host`` from pinned host
buffers (copies inside the timed region).  ``cpu_baseline`` times the CPU
oracle on the host cores over every pair of the workload at every
threshold, and ``parity`` compares its decisions with the GPU's, pair by
pair.

``--impl reference`` times the CPU oracle alone on the same workload (the
reference arm).  Under torchrun each rank filters its own 30M pairs (weak
scaling, no collective on the data path).
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import re
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

N_PAIRS = 30_000_000
M = 100
SWEEP = [0, 2, 4, 6, 8, 10]
# the step's filter launches, as ss_filter_sweep makes them: the sweep's
# thresholds up to 4 share one pass over the pairs (their walks cost less
# than the pass), every other threshold has its own launch
SHARED_MAX_E = 4


def sweep_groups(sweep):
    low = [e for e in sweep if e <= SHARED_MAX_E]
    groups = [tuple(low)] if len(low) >= 2 else [(e,) for e in low]
    return groups + [(e,) for e in sweep if e > SHARED_MAX_E]


GROUPS = sweep_groups(SWEEP)
SEED = 1910_09020 + 2
WORKLOAD = ("short-read threshold sweep: 30M synthetic pairs x 100 bp "
            "(even pairs Poisson(3) edits, odd pairs random), "
            "E in {0,2,4,6,8,10}, plain form (one sweep call: a shared pass "
            "for E <= 4, one launch per larger E)")
METRIC = "sequence pairs/sec (and Gbases/s) per GB300 vs roofline"
# algorithmic bytes of one pair decision: both sequences at 2 bits per base
# plus the accept byte and the int32 obstacle count
FILTER_BYTES_PER_PAIR = 2 * ((M + 3) // 4) + 1 + 4
# pack: both sequences read as ASCII, written at 2 bits per base
PACK_BYTES_PER_PAIR = 2 * M + 2 * ((M + 3) // 4)
# op model of the method per the lazy maze of Section 2.4, in two
# formulations of the same greedy; the roofline takes the cheaper one for
# each threshold (the method's work is what its cheapest evaluation needs):
# * row words: per evaluated 32-column row word 7 logic/shift ops + 1
#   find-first; per iteration one max per row plus 4 bookkeeping ops;
# * columns: per column walked, ceil((2E+1)/32) words holding its 2E+1
#   rows, each 7 ops (2 funnel shifts of the query planes, 2 XORs with the
#   broadcast reference base, 1 OR, 1 AND into the surviving rows, 1 for
#   the broadcast); per iteration 4 bookkeeping ops; no find-first.
# * bit-sliced columns: 32 pairs of one length walked together, one pair
#   per bit; per column and 32 pairs two three-input logic ops per row (the
#   two code bits' equality), E three-input ORs for the column's "all rows
#   dead" and E+1 ops of the saturating count: (6E+3)/32 logic ops per pair
#   and column, over all m columns (a group of 32 stops early only when all
#   of its pairs are past E).  The S_d | z restarts are adds on the FMA pipe
#   and are not counted against the logic pipe.
K_WORD, K_RED, K_ITER = 7, 1, 4
K_COL = 7


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=60)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--pairs", type=int, default=N_PAIRS,
                    help="pairs per GPU (default: the full workload)")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--headline-only", action="store_true",
                    help="skip the batched and served forms")
    ap.add_argument("--workload", default="all",
                    choices=["all", "batched", "long", "two_lengths"],
                    help="long: only pairs of one index class (profiling); "
                         "batched: only the persistent launch of the uneven "
                         "batch (for profiling); two_lengths: only the "
                         "two-length comparison of forms")
    ap.add_argument("--serve-seconds", type=float, default=4.0,
                    help="arrival window of each offered load")
    ap.add_argument("--batched-pairs", type=int, default=2_000_000,
                    help="pairs of the uneven batch")
    ap.add_argument("--details", default=DETAILS, metavar="FILE",
                    help="file for the whole record, of which the printed "
                         "line holds the short values")
    return ap.parse_args()


# ---- distributed plumbing ----------------------------------------------------

def dist_setup():
    import torch
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    else:
        torch.cuda.set_device(local)
    return rank, world, local


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def max_over_ranks(x: float, world: int) -> float:
    if world == 1:
        return x
    import torch
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64, device="cuda")
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


# ---- clocks --------------------------------------------------------------------

class ClockSampler:
    """nvidia-smi samples of SM clock and throttle reasons during a region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,"
              "clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")

    def __init__(self, device: int):
        self.device = device
        self.proc = None
        self.path = None

    def start(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.device),
                 f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "100"],
                stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None
        time.sleep(0.3)

    def stop(self) -> dict:
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": [],
                    "samples": 0}
        time.sleep(0.15)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        rows = []
        for line in open(self.path):
            parts = [p.strip() for p in line.split(",")]
            if len(parts) >= 9:
                rows.append(parts)
        os.unlink(self.path)
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown",
                 "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4)
                          if r[5 + i].lower().startswith("active")})
        return {"sm_mhz": float(np.median(sm)) if sm else None,
                "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(rows)}


# ---- peaks ---------------------------------------------------------------------

def measured_peaks() -> dict:
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        d = json.load(open(path))
        return {"hbm_gbs": float(d["hbm_gbs"]), "hbm_source": "measured"}
    return {"hbm_gbs": 6800.0, "hbm_source": "fallback"}


# the source files each profiled kernel is compiled from: a change to any of
# them makes its committed DRAM-traffic figure stale
KERNEL_SOURCES = {
    "k_rw_uniform": ["ss_device.cuh", "ss_rw_config.h", "ss_rw.cuh",
                     "ss_rwc.cuh", "ss_rw_launch.cuh", "ss_rw_e0.cu",
                     "ss_rw_e1.cu", "ss_rw_e2.cu", "ss_rw_e3.cu"],
    "k_pack_fixed": ["ss_device.cuh", "ss_pack.cuh", "ss_pack.cu"],
    "k_sliced": ["ss_device.cuh", "ss_rw_config.h", "ss_sliced.cuh",
                 "ss_sliced.cu"],
    "k_sliced_set": ["ss_device.cuh", "ss_rw_config.h", "ss_sliced.cuh",
                     "ss_sliced_set.cu"],
    "k_pack_sliced_span": ["ss_device.cuh", "ss_rw_config.h", "ss_pack.cuh",
                           "ss_sliced.cuh", "ss_pack.cu"],
}


def code_of(text: str) -> str:
    """C/CUDA source without comments and blank space: what compiles."""
    text = re.sub(r"/\*.*?\*/", " ", text, flags=re.S)
    text = re.sub(r"//[^\n]*", " ", text)
    return " ".join(text.split())


def kernel_source_hash(kernel: str) -> str:
    """Hash of the code (comments and layout ignored) a profiled kernel is
    compiled from."""
    h = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_1910_09020_gb300", "csrc")
    for name in KERNEL_SOURCES[kernel]:
        with open(os.path.join(csrc, name)) as f:
            h.update(code_of(f.read()).encode())
    return h.hexdigest()[:16]


def ncu_traffic(kernel: str) -> float | None:
    """DRAM bytes per pair of a kernel from the committed ncu summary, or
    None if the kernels changed since it was captured."""
    path = os.path.join(ROOT, "profiles", "traffic.json")
    if not os.path.exists(path):
        return None
    d = json.load(open(path))
    k = d.get("kernels", {}).get(kernel)
    if k is None or k.get("source_sha") != kernel_source_hash(kernel):
        return None
    return float(k["dram_bytes_per_pair"])


# ---- CPU oracle (baseline leg and reference arm) --------------------------------

def oracle_sample(n: int, first: int = 0):
    from paper_1910_09020_gb300 import synth
    return synth.pairs_fixed(SEED, first, n, M, synth.SHORT_POISSON)


def time_oracle(reads, refs, threads: int = 0):
    """Oracle over every threshold of the sweep; returns (seconds, per-E
    stats (cells, words, iterations, columns) summed over pairs)."""
    import oracle
    stats = {}
    t0 = time.perf_counter()
    for E in SWEEP:
        _, _, st = oracle.filter_batch(reads, refs, M, E, threads=threads,
                                       with_stats=True)
        stats[E] = st
    return time.perf_counter() - t0, stats


def cpu_oracle_full(reads, refs, acc, obs):
    """The oracle over EVERY pair of the workload at every threshold of the
    sweep (about 9 s on 16 host cores at 30M pairs): its time is the CPU
    baseline, its counters feed the op model, and its decisions are compared
    element by element with the GPU's (acc, obs: host arrays [E, n]).
    Returns (cpu_baseline, per-E stats, parity)."""
    import oracle
    cores = oracle.default_threads()
    n = reads.shape[0]
    stats = {}
    t_all = 0.0
    mismatches = 0
    first_bad = None
    for t, E in enumerate(SWEEP):
        t0 = time.perf_counter()
        oa, oo, st = oracle.filter_batch(reads, refs, M, E, with_stats=True)
        t_all += time.perf_counter() - t0
        stats[E] = st
        bad = np.flatnonzero((oa != acc[t]) | (oo != obs[t]))
        mismatches += int(len(bad))
        if len(bad) and first_bad is None:
            first_bad = {"E": E, "pair": int(bad[0]),
                         "gpu": [int(acc[t][bad[0]]), int(obs[t][bad[0]])],
                         "oracle": [int(oa[bad[0]]), int(oo[bad[0]])]}
    cpu = {"value": n * len(SWEEP) / t_all, "unit": "pairs/s",
           "cores": cores, "kind": "oracle",
           "sample": f"every pair of the workload ({n}) x {len(SWEEP)} "
                     f"thresholds ({t_all:.1f} s, {cores} host threads)"}
    parity = {"pairs_checked": n, "decisions_checked": n * len(SWEEP),
              "mismatches": mismatches, "first_mismatch": first_bad,
              "against": "CPU oracle (Eq. 1, Section 2.4 steps 1-5), "
                         "accept flag and obstacle count of every pair"}
    return cpu, stats, parity


def row_word_ops(E: int, words, iters):
    """ALU ops of the row-word formulation (and `words` find-first ops)."""
    return words * K_WORD + iters * (2 * E + 1) * K_RED + iters * K_ITER


def column_ops(E: int, iters, cols):
    """ALU ops of the column formulation (no find-first)."""
    return cols * ((2 * E + 1 + 31) // 32) * K_COL + iters * K_ITER


def sliced_ops(E: int, m: int, n: int):
    """ALU ops of the bit-sliced column formulation for n pairs of length m
    (every column walked)."""
    return n * m * (6 * E + 3) / 32


def model_ops(E: int, words, iters, cols, sliced=None):
    """ALU and find-first ops of the cheapest formulation (see K_COL), and
    which one it is.  sliced: the bit-sliced formulation's ops where the
    pairs come in groups of one length (else not a candidate)."""
    rows = row_word_ops(E, words, iters)
    by_col = column_ops(E, iters, cols)
    best = (rows, words, "row words")
    if by_col < best[0]:
        best = (by_col, 0, "columns")
    if sliced is not None and sliced < best[0]:
        best = (sliced, 0, "bit-sliced columns")
    return best


def op_model(stats: dict, n: int, m: int | None = None) -> dict:
    """Per-pair algorithmic ALU and find-first ops of each threshold (with
    m: the bit-sliced formulation is a candidate, uniform length m)."""
    out = {}
    for E, (cells, words, iters, cols) in stats.items():
        sl = sliced_ops(E, m, n) if m else None
        alu, xu, form = model_ops(E, words, iters, cols, sl)
        out[E] = {"alu_ops_per_pair": alu / n, "xu_ops_per_pair": xu / n,
                  "model": form,
                  "alu_ops_row_words_per_pair":
                      row_word_ops(E, words, iters) / n,
                  "alu_ops_columns_per_pair": column_ops(E, iters, cols) / n,
                  "iterations_per_pair": iters / n,
                  "columns_per_pair": cols / n,
                  "cells_per_pair": cells / n}
        if sl is not None:
            out[E]["alu_ops_sliced_per_pair"] = sl / n
    return out


# ---- reference arm ----------------------------------------------------------------

def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    import oracle
    cores = oracle.default_threads()
    r, f = oracle_sample(20000)
    dt, _ = time_oracle(r, f)
    per_step_s = 1.5
    total_budget = 150.0
    steps_total = args.steps + args.warmup
    per_step_s = min(per_step_s, total_budget / max(steps_total, 1))
    n = int(max(2000, 20000 * per_step_s / max(dt, 1e-6)))
    times = []
    for s in range(steps_total):
        rr, ff = oracle_sample(n, first=s * n)
        dt, _ = time_oracle(rr, ff)
        if s >= args.warmup:
            times.append(dt)
    t = float(np.sum(times))
    value = n * len(SWEEP) * len(times) / t
    line = {
        "impl": "reference", "metric": METRIC, "value": value,
        "unit": "pairs/s", "n_gpus": args.gpus, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": 1e3 * t / len(times),
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "u8", "data": "synthetic",
        # the workload this arm stands in for (the GPU arm's config); the
        # bounded sample actually timed is stated in cpu_baseline.sample
        "config": config_dict(args.gpus, n_override=args.pairs),
        "cpu_baseline": {"value": value, "unit": "pairs/s", "cores": cores,
                         "kind": "oracle",
                         "sample": f"step s (warm-up first) times pairs "
                                   f"s*{n} .. (s+1)*{n}-1 of the workload "
                                   f"x {len(SWEEP)} thresholds, {cores} "
                                   f"host threads"},
        "e2e": {"value": value, "unit": "pairs/s", "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
        # what one timed step holds: ms_per_step is the time of this many
        # pairs (a slice of the config's pairs_per_gpu), not of the config
        "sample_pairs_per_step": n,
        "sample_decisions_per_step": n * len(SWEEP),
        "ms_per_config_step": 1e3 * t / len(times) * (args.pairs / n),
    }
    print(json.dumps(line), flush=True)
    return 0


# Longest value (as JSON) that the printed line carries of its own: the whole
# record was some 26 KB, longer than what a caller keeps of a program's
# output, and could not be read back.
LINE_VALUE_CHARS = 800
DETAILS = os.path.join(ROOT, "paper_1910_09020_gb300", "_build",
                       "bench_details.json")


def short_line(line: dict, details: str | None) -> dict:
    """The record without its long values (of a long section its numbers);
    `details` is the file that holds all of it."""
    out = {}
    for k, v in line.items():
        if len(json.dumps(v)) > LINE_VALUE_CHARS and isinstance(v, dict):
            v = {x: y for x, y in v.items()
                 if isinstance(y, (bool, int, float))}
        if v != {} and len(json.dumps(v)) <= LINE_VALUE_CHARS:
            out[k] = v
    if details:
        out["details"] = os.path.relpath(details, ROOT)
    return out


def print_line(line: dict, path: str) -> None:
    """One JSON line on stdout, the whole record in the file `path`."""
    try:
        os.makedirs(os.path.dirname(os.path.abspath(path)), exist_ok=True)
        with open(path, "w") as f:
            json.dump(line, f)
            f.write("\n")
    except OSError as err:
        print(f"bench: {path} not written: {err}", file=sys.stderr)
        path = None
    print(json.dumps(short_line(line, path)), flush=True)


def config_dict(world: int, n_override: int | None = None) -> dict:
    return {"workload": WORKLOAD, "pairs_per_gpu": n_override or N_PAIRS,
            "read_length": M, "thresholds": SWEEP, "format": "ASCII resident, "
            "packed in the step to 2 bits per base, bit-sliced (32 pairs per "
            "word)", "parallelism": f"replicas x{world}",
            "l2": "inputs larger than L2 (6 GB ASCII + 1.5 GB packed)"}


# ---- batched and served forms (configurations beside the headline) ------------

def _ev():
    import torch
    return torch.cuda.Event(enable_timing=True)


def _time_ms(fn, reps: int, sync) -> float:
    import torch
    fn()
    sync()
    torch.cuda.synchronize()
    a, z = _ev(), _ev()
    a.record()
    for _ in range(reps):
        fn()
    z.record()
    torch.cuda.synchronize()
    sync()
    return a.elapsed_time(z) / reps


def _pack_varlen(F, L, recipe, seed):
    """Pairs of lengths L, generated and packed on the device; returns the
    device packed buffers, word offsets, lengths and host byte offsets."""
    import torch

    from paper_1910_09020_gb300 import synth
    reads, refs, off = synth.pairs_varlen(seed, 0, L, recipe)
    words = (L.astype(np.int64) + 15) // 16
    woff = np.zeros(len(L) + 1, np.int64)
    np.cumsum(words, out=woff[1:])
    dL = torch.from_numpy(L).cuda()
    dwo = torch.from_numpy(woff[:-1].copy()).cuda()
    doff = torch.from_numpy(off[:-1].copy()).cuda()
    pq = torch.empty(int(woff[-1]), dtype=torch.int32, device="cuda")
    pr = torch.empty_like(pq)
    dq = torch.from_numpy(reads).cuda()
    F.pack(dq, offsets=doff, lengths=dL, out=pq, out_offsets=dwo)
    del dq
    dr = torch.from_numpy(refs).cuda()
    F.pack(dr, offsets=doff, lengths=dL, out=pr, out_offsets=dwo)
    del dr
    F.sync()
    return pq, pr, dwo, dL, woff, (reads, refs, off)


def _oracle_model(host, L, E, idx):
    """Oracle time and the op model (per threshold group, the cheaper of
    the row-word and column formulations) on a sample of pairs.  Returns
    (seconds, alu ops, xu ops, cells)."""
    from concurrent.futures import ThreadPoolExecutor

    import oracle
    reads, refs, off = host

    def group(e):
        # one threshold group on one host thread (the oracle's call
        # releases the interpreter, so groups run side by side)
        sel = idx[E[idx] == e]
        sub_r = np.concatenate([reads[off[i]:off[i] + L[i]] for i in sel])
        sub_f = np.concatenate([refs[off[i]:off[i] + L[i]] for i in sel])
        so = np.zeros(len(sel) + 1, np.int64)
        np.cumsum(L[sel], out=so[1:])
        _, _, (c, w, it, col) = oracle.filter_batch(sub_r, sub_f, L[sel],
                                                    E[sel], offsets=so,
                                                    threads=1,
                                                    with_stats=True)
        a_, x_, _ = model_ops(int(e), w, it, col)  # the cheaper form
        return a_, x_, c

    t0 = time.perf_counter()
    groups = np.unique(E[idx])
    with ThreadPoolExecutor(oracle.default_threads()) as ex:
        res = list(ex.map(group, groups[::-1]))  # largest E first
    t = time.perf_counter() - t0
    alu = sum(r[0] for r in res)
    xu = sum(r[1] for r in res)
    cells = sum(r[2] for r in res)
    return t, alu, xu, cells


def run_batched(F, ipk, hbm_gbs, want_cpu: bool,
                per_length_too: bool = True, n: int = 2_000_000) -> dict:
    """Uneven batch of 2M pairs, lengths log-uniform 64..10000, edit rate
    U[0, 0.10], E = 5 % of each length: one bucketed persistent launch
    (CUDA graph, autotuned) against one launch per distinct length."""
    import torch

    from paper_1910_09020_gb300 import binding, synth
    seed = 1910_09020 + 4
    L = np.sort(synth.log_uniform(seed, 0, n, 64, 10000)).astype(np.int32)
    E = synth.thresholds(L, 5)
    pq, pr, dwo, dL, woff, host = _pack_varlen(F, L, synth.rate_recipe(0.10),
                                               seed)
    dE = torch.from_numpy(E).cuda()
    acc = torch.empty(n, dtype=torch.uint8, device="cuda")
    obs = torch.empty(n, dtype=torch.int32, device="cuda")
    rmax, k, _ = F.autotune(pq, pr, offsets=dwo, lengths=dL, E=dE, reps=2,
                            out_accept=acc, out_obstacles=obs)
    persistent = lambda: F.filter(pq, pr, offsets=dwo, lengths=dL, E=dE,
                                  out_accept=acc, out_obstacles=obs)
    t_p = _time_ms(persistent, 10, F.sync)
    # the same batch without the persistent form: pairs are sorted by
    # length, so each distinct length the plain kernel covers (E <= 31,
    # m <= 1024) is one fixed-stride plain launch over the same packed
    # buffers; the pairs it does not cover (the longer ones, E > 31) can
    # only go through one bucketed call of their own
    plain_ok = (E <= binding.PLAIN_MAX_E) & (L <= binding.PLAIN_MAX_M)
    k_tail = int(np.argmin(plain_ok)) if not plain_ok.all() else n
    assert plain_ok[:k_tail].all() and not plain_ok[k_tail:].any()
    starts = np.flatnonzero(np.r_[True, L[1:k_tail] != L[:k_tail - 1]])
    ends = np.r_[starts[1:], k_tail]
    acc2 = torch.empty_like(acc)
    obs2 = torch.empty_like(obs)

    def per_class_plain():
        for a, b in zip(starts, ends):
            F.filter(pq[int(woff[a]):], pr[int(woff[a]):], m=int(L[a]),
                     e=int(E[a]), n=int(b - a), out_accept=acc2[a:b],
                     out_obstacles=obs2[a:b])
        if k_tail < n:
            F.filter(pq, pr, offsets=dwo[k_tail:], lengths=dL[k_tail:],
                     E=dE[k_tail:], out_accept=acc2[k_tail:],
                     out_obstacles=obs2[k_tail:])
    if not per_length_too:
        return {"persistent_graph_ms": t_p, "pairs": n}
    t_l = _time_ms(per_class_plain, 5, F.sync)
    same = bool(torch.equal(acc, acc2) and torch.equal(obs, obs2))
    bases = int(L.sum())
    bytes_alg = float(np.sum(2 * ((L.astype(np.int64) + 3) // 4) + 5 + 16))
    out = {
        "workload": "2M pairs, lengths log-uniform 64..10000 bp, edit rate "
                    "U[0,0.10] (80 % substitutions), E = 5 % of length",
        "pairs": n, "bases": bases,
        "persistent_graph": {"ms": t_p, "pairs_per_s": n / (t_p * 1e-3),
                             "gbases_per_s": bases / (t_p * 1e-3) / 1e9,
                             "tuning": {"rw_max_e": rmax, "cw_subgrid": k}},
        "per_class_plain": {
            "ms": t_l, "pairs_per_s": n / (t_l * 1e-3),
            "plain_launches": int(len(starts)), "plain_pairs": k_tail,
            "bucketed_tail_pairs": n - k_tail,
            "form": "one plain launch per distinct length with E <= 31 and "
                    "m <= 1024, one bucketed call for the longer pairs"},
        "per_class_plain_over_persistent": t_l / t_p,
        "results_identical": same,
        "accept_rate": float(acc.float().mean().item()),
    }
    # accuracy of every decision against the warp-per-pair banded verifier
    # (E <= 511 covers the whole batch), outside the timed region
    a, b = _ev(), _ev()
    a.record()
    ed = F.edit_distance_varlen(pq, pr, dwo, dL, dE)
    b.record()
    F.sync()
    close = ed <= dE
    accd = acc.bool()
    fa = int((accd & ~close).sum().item())
    fr = int((~accd & close).sum().item())
    tr = int((~accd & ~close).sum().item())
    out["accuracy"] = {"false_accepts": fa, "false_rejects": fr,
                       "false_accept_rate": fa / max(fa + tr, 1),
                       "verifier_ms": a.elapsed_time(b)}
    t_hbm = bytes_alg / (hbm_gbs * 1e9)
    roof = {"t_hbm_ms": 1e3 * t_hbm, "algorithmic_bytes": bytes_alg}
    if want_cpu:
        rng = np.random.default_rng(seed)
        idx = np.sort(rng.choice(n, 20000, replace=False))
        t_o, alu, xu, cells = _oracle_model(host, L, E, idx)
        scale = n / len(idx)
        t_alu = alu * scale / ipk["lop3"]
        t_xu = xu * scale / ipk["bfind"]
        roof.update({"t_alu_ms": 1e3 * t_alu, "t_xu_ms": 1e3 * t_xu,
                     "alu_ops_per_pair": alu / len(idx),
                     "cells_per_pair": cells / len(idx)})
        import oracle
        out["cpu_baseline"] = {
            "value": len(idx) / t_o, "unit": "pairs/s", "kind": "oracle",
            "cores": oracle.default_threads(),
            "sample": f"{len(idx)} pairs drawn uniformly from the batch "
                      f"({t_o:.1f} s)"}
    t_bound = max(roof.get("t_alu_ms", 0), roof.get("t_xu_ms", 0),
                  roof["t_hbm_ms"])
    roof["bound"] = ("hbm" if t_bound == roof["t_hbm_ms"] else
                     "alu" if t_bound == roof.get("t_alu_ms") else "xu")
    roof["frac"] = t_bound / t_p
    roof["note"] = ("ALU term: per threshold group the cheaper of the "
                    "row-word and column op models of the lazy maze; the "
                    "warp/CTA kernels evaluate each 32-row word only until "
                    "its rows die, so they can run below either model")
    out["roofline"] = roof
    del pq, pr
    return out


def _fixed_model(reads, refs, m, E):
    """Op model (the cheapest formulation, see K_COL; the pairs share one
    length, so the bit-sliced one is a candidate) of fixed-length pairs:
    per-pair ALU and find-first ops from the oracle's counters."""
    import oracle
    n = len(reads)
    _, _, (_, w, it, col) = oracle.filter_batch(reads, refs, m, E,
                                                with_stats=True)
    alu, xu, _ = model_ops(E, w, it, col, sliced_ops(E, m, n))
    return alu / n, xu / n


def run_two_lengths(F, ipk=None, hbm_gbs=None, sample=20000) -> dict:
    """10M pairs of 250 bp and 10M of 150 bp, edit rate U[0, 0.12], E = 0 %
    .. 10 % of length: two plain launches (pair-major packed input, as the
    persistent graph reads) against one persistent graph; over the
    bit-sliced layout, the two plain launches one after the other against
    one segmented call (ss_filter_segments: a replayed CUDA graph whose two
    launches run side by side); each with its roofline fraction (HBM bytes
    of the form; ALU ops of the cheapest op model, the bit-sliced one
    included, from the oracle's counters on `sample` pairs of each
    length)."""
    import torch

    from paper_1910_09020_gb300 import synth
    n3 = 10_000_000
    seed = 1910_09020 + 3
    rec = synth.rate_recipe(0.12)
    from paper_1910_09020_gb300 import binding
    samples = {}
    bufs = []
    sbufs = []  # the same pairs in the bit-sliced layout
    for m, first in ((250, 0), (150, n3)):
        r, f = synth.pairs_fixed(seed, first, n3, m, rec)
        samples[m] = (r[:sample].copy(), f[:sample].copy())
        dr_, df_ = (torch.from_numpy(r.reshape(-1)).cuda(),
                    torch.from_numpy(f.reshape(-1)).cuda())
        q = F.pack(dr_, m=m, n=n3)
        g = F.pack(df_, m=m, n=n3)
        sbufs.append((F.pack_sliced(dr_, m=m, n=n3),
                      F.pack_sliced(df_, m=m, n=n3)))
        F.sync()
        bufs.append((q, g))
        del r, f, dr_, df_
    w250, w150 = 16, 10
    allq = torch.cat([bufs[0][0], bufs[1][0]])
    allr = torch.cat([bufs[0][1], bufs[1][1]])
    offs = torch.cat([torch.arange(n3, dtype=torch.int64) * w250,
                      n3 * w250 + torch.arange(n3, dtype=torch.int64) * w150]
                     ).cuda()
    lens = torch.cat([torch.full((n3,), 250, dtype=torch.int32),
                      torch.full((n3,), 150, dtype=torch.int32)]).cuda()
    a = torch.empty(2 * n3, dtype=torch.uint8, device="cuda")
    o = torch.empty(2 * n3, dtype=torch.int32, device="cuda")
    a2, o2 = torch.empty_like(a), torch.empty_like(o)
    a3, o3 = torch.empty_like(a), torch.empty_like(o)
    a4, o4 = torch.empty_like(a), torch.empty_like(o)
    rows = []
    same = True
    for pct in range(0, 11):
        e250, e150 = 250 * pct // 100, 150 * pct // 100
        Es = torch.cat([torch.full((n3,), e250, dtype=torch.int32),
                        torch.full((n3,), e150, dtype=torch.int32)]).cuda()

        def plain():
            F.filter(bufs[0][0], bufs[0][1], m=250, e=e250, n=n3,
                     out_accept=a[:n3], out_obstacles=o[:n3])
            F.filter(bufs[1][0], bufs[1][1], m=150, e=e150, n=n3,
                     out_accept=a[n3:], out_obstacles=o[n3:])
        persistent = lambda: F.filter(allq, allr, offsets=offs, lengths=lens,
                                      E=Es, out_accept=a2, out_obstacles=o2)

        def plain_sliced():
            F.filter(sbufs[0][0], sbufs[0][1], m=250, e=e250, n=n3,
                     fmt=binding.SS_FMT_SLICED2, out_accept=a3[:n3],
                     out_obstacles=o3[:n3])
            F.filter(sbufs[1][0], sbufs[1][1], m=150, e=e150, n=n3,
                     fmt=binding.SS_FMT_SLICED2, out_accept=a3[n3:],
                     out_obstacles=o3[n3:])
        def graph_sliced():
            F.filter_segments(
                [(sbufs[0][0], sbufs[0][1], 250, e250, n3,
                  (a4[:n3], o4[:n3])),
                 (sbufs[1][0], sbufs[1][1], 150, e150, n3,
                  (a4[n3:], o4[n3:]))], fmt=binding.SS_FMT_SLICED2)
        tp = _time_ms(plain, 5, F.sync)
        tb = _time_ms(persistent, 5, F.sync)
        ts = _time_ms(plain_sliced, 5, F.sync)
        tg = _time_ms(graph_sliced, 5, F.sync)
        same &= bool(torch.equal(a, a2) and torch.equal(o, o2) and
                     torch.equal(a, a3) and torch.equal(o, o3) and
                     torch.equal(a, a4) and torch.equal(o, o4))
        # accuracy of these decisions against the banded edit distance
        conf = [0, 0, 0, 0]
        for (q, g), (m, e), sl in (((bufs[0]), (250, e250), slice(0, n3)),
                                    ((bufs[1]), (150, e150),
                                     slice(n3, 2 * n3))):
            ed = F.edit_distance(q, g, m=m, e=e, n=n3)
            for k, v in enumerate(F.confusion(a[sl], ed, e=e)):
                conf[k] += v
        ta, fa, fr, tr = conf
        row = {"E_pct": pct, "E": [e250, e150],
               "plain_pairs_per_s": 2 * n3 / (tp * 1e-3),
               "persistent_pairs_per_s": 2 * n3 / (tb * 1e-3),
               "plain_ms": tp, "persistent_ms": tb,
               "plain_sliced_ms": ts,
               "plain_sliced_pairs_per_s": 2 * n3 / (ts * 1e-3),
               "graph_sliced_ms": tg,
               "graph_sliced_pairs_per_s": 2 * n3 / (tg * 1e-3),
               "false_accepts": fa, "false_rejects": fr,
               "false_accept_rate": fa / max(fa + tr, 1)}
        if ipk and hbm_gbs:
            # algorithmic bytes: both packed sequences and the results; the
            # persistent form also reads each pair's offset, length and E
            b_plain = n3 * (2 * ((250 + 3) // 4) + 5 + 2 * ((150 + 3) // 4)
                            + 5)
            b_pers = b_plain + 2 * n3 * 16
            alu = xu = 0.0
            for m, e in ((250, e250), (150, e150)):
                a_, x_ = _fixed_model(*samples[m], m, e)
                alu += a_ * n3
                xu += x_ * n3
            t_alu = 1e3 * alu / ipk["lop3"]
            t_xu = 1e3 * xu / ipk["bfind"]
            for form, nb, ms in (("plain", b_plain, tp),
                                 ("persistent", b_pers, tb),
                                 ("plain_sliced", b_plain, ts),
                                 ("graph_sliced", b_plain, tg)):
                t_hbm = 1e3 * nb / (hbm_gbs * 1e9)
                t = max(t_hbm, t_alu, t_xu)
                row[form + "_roofline"] = {
                    "bound": "hbm" if t == t_hbm else
                             "alu" if t == t_alu else "xu",
                    "t_hbm_ms": t_hbm, "t_alu_ms": t_alu, "t_xu_ms": t_xu,
                    "frac": t / ms}
        rows.append(row)
    return {"workload": "10M x 250 bp + 10M x 150 bp, edit rate U[0,0.12], "
                        "E = 0..10 % of length",
            "roofline_note": "max(HBM, ALU, find-first) time of the form / "
                             "measured time; ALU from the cheapest op model "
                             "(row words, columns, bit-sliced columns) "
                             f"on {sample} pairs of each length",
            "per_E": rows, "results_identical": same}


def run_submaze(F, sq, sr, pq, pr, n, acc, obs, t=8, y=3) -> dict:
    """Snake-on-Chip's sub-maze mode (t=8 columns, y=3 segments each, the
    hardware design point of Section 2.5) on the headline pairs, over the
    bit-sliced layout (and, beside it, the pair-major one): per-E launch
    time and the decisions it adds over the exact filter just timed."""
    import torch

    from paper_1910_09020_gb300 import binding

    def timed(f):
        f()  # warm
        a, b = _ev(), _ev()
        a.record()
        reps = 5
        for _ in range(reps):
            r = f()
        b.record()
        torch.cuda.synchronize()
        return a.elapsed_time(b) / reps, r

    out = []
    for k, E in enumerate(SWEEP):
        ms, (sacc, sobs) = timed(lambda: F.filter_submaze(
            sq, sr, m=M, e=E, t=t, y=y, n=n, fmt=binding.SS_FMT_SLICED2))
        pm_ms, (pacc, pobs) = timed(lambda: F.filter_submaze(
            pq, pr, m=M, e=E, t=t, y=y, n=n))
        same = bool(torch.equal(sacc, pacc) and torch.equal(sobs, pobs))
        extra = int((sacc.to(torch.int32) - acc[k].to(torch.int32)).clamp(min=0)
                    .sum().item())
        lost = int((acc[k].to(torch.int32) - sacc.to(torch.int32)).clamp(min=0)
                   .sum().item())
        above = int((sobs > obs[k]).sum().item())
        gbs = n * FILTER_BYTES_PER_PAIR / (ms * 1e-3) / 1e9
        out.append({"E": E, "ms": ms, "pairs_per_s": n / (ms * 1e-3),
                    "hbm_gbs": gbs,
                    "hbm_frac": gbs / measured_peaks()["hbm_gbs"],
                    "pair_major_ms": pm_ms, "forms_identical": same,
                    "accepts": int(sacc.sum(dtype=torch.int64).item()),
                    "exact_accepts": int(acc[k].sum(dtype=torch.int64).item()),
                    "added_accepts": extra, "lost_accepts": lost,
                    "count_above_exact": above})
    return {"t": t, "y": y, "pairs": n, "form": "bit-sliced (k_sliced_sub)",
            "per_E": out}


def run_unequal(F, n=2_000_000) -> dict:
    """Reads of 100 bp against reference windows of 92..116 bp (the read
    inside random flanks, or the window cut short): the filter for pairs of
    different lengths, one launch per E over the pair-major layout; and the
    same pairs bucketed by window length into 25 uniform segments over the
    bit-sliced layout, one segmented call per E (results checked equal).
    Beside them, the plain sliced launch on 2M pairs of equal length."""
    import torch

    from paper_1910_09020_gb300 import binding, synth
    data = synth.pairs_unequal(SEED + 7, 0, n, M, synth.SHORT_POISSON, -8, 16)
    reads, ro, rl, refs, fo, fl = data
    dev = torch.device("cuda", torch.cuda.current_device())

    def packed(ascii_, off, lens):
        words = (lens.astype(np.int64) + 15) // 16
        woff = np.zeros(len(lens) + 1, np.int64)
        np.cumsum(words, out=woff[1:])
        out = torch.zeros(int(woff[-1]) + 4, dtype=torch.int32, device=dev)
        F.pack(torch.from_numpy(ascii_).to(dev),
               offsets=torch.from_numpy(off[:-1].astype(np.int64)).to(dev),
               lengths=torch.from_numpy(lens.astype(np.int32)).to(dev),
               out=out, out_offsets=torch.from_numpy(woff[:-1]).to(dev))
        return out, torch.from_numpy(woff[:-1]).to(dev)

    q, qo = packed(reads, ro, rl)
    r, fo_d = packed(refs, fo, fl)
    ql = torch.from_numpy(rl.astype(np.int32)).to(dev)
    rlen = torch.from_numpy(fl.astype(np.int32)).to(dev)
    # the bit-sliced segments: pairs grouped by window length (host-side
    # bucketing of the generator's output, outside the timed region)
    order = np.argsort(fl, kind="stable")
    rd = reads.reshape(n, M)
    segs = []
    for L in np.unique(fl):
        idx = order[fl[order] == L]
        rows = refs[(fo[idx][:, None] + np.arange(L)[None, :]).reshape(-1)]
        sq = F.pack_sliced(torch.from_numpy(
            np.ascontiguousarray(rd[idx]).reshape(-1)).to(dev), m=M,
            n=len(idx))
        sr = F.pack_sliced(torch.from_numpy(rows).to(dev), m=int(L),
                           n=len(idx))
        a_ = torch.empty(len(idx), dtype=torch.uint8, device=dev)
        o_ = torch.empty(len(idx), dtype=torch.int32, device=dev)
        segs.append([sq, sr, (M, int(L)), 0, len(idx), (a_, o_),
                     torch.from_numpy(idx).to(dev)])
    # equal-length pairs of the same recipe for the plain sliced launch
    er, ef = synth.pairs_fixed(SEED + 8, 0, n, M, synth.SHORT_POISSON)
    eq_q = F.pack_sliced(torch.from_numpy(er.reshape(-1)).to(dev), m=M, n=n)
    eq_r = F.pack_sliced(torch.from_numpy(ef.reshape(-1)).to(dev), m=M, n=n)
    del er, ef
    F.sync()
    # algorithmic bytes per launch: both packed sequences, their word
    # offsets and lengths (8 + 4 B each), and the two results
    words = int(((rl.astype(np.int64) + 15) // 16).sum()
                + ((fl.astype(np.int64) + 15) // 16).sum())
    nbytes = 4 * words + n * (2 * 12 + 5)
    sliced_bytes = int(n * ((M + 3) // 4) + ((fl.astype(np.int64) + 3)
                                             // 4).sum() + 5 * n)
    out = []
    same = True
    for E in (2, 6, 10):
        F.filter_unequal(q, qo, ql, r, fo_d, rlen, e=E)
        a, b = _ev(), _ev()
        a.record()
        reps = 5
        for _ in range(reps):
            acc, obs = F.filter_unequal(q, qo, ql, r, fo_d, rlen, e=E)
        b.record()
        torch.cuda.synchronize()
        ms = a.elapsed_time(b) / reps
        gbs = nbytes / (ms * 1e-3) / 1e9
        # the segment table built once and handed to the C call directly
        # (what a caller of the library does; the Python wrapper would add
        # its per-segment checks to every call)
        arr = (binding.Segment * len(segs))()
        for i, sg in enumerate(segs):
            arr[i] = binding.Segment(sg[0].data_ptr(), sg[1].data_ptr(),
                                     sg[4], M, E, sg[5][0].data_ptr(),
                                     sg[5][1].data_ptr(), sg[2][1])
        stream = torch.cuda.current_stream().cuda_stream

        def seg_call():
            rc = binding.ss_filter_segments(F.ctx, arr, len(segs),
                                            binding.SS_FMT_SLICED2, 0, stream)
            assert rc == binding.SS_OK, rc
        ms_s = _time_ms(seg_call, reps, F.sync)
        for sg in segs:  # back to the batch's order
            same &= bool(torch.equal(sg[5][0], acc[sg[6]]) and
                         torch.equal(sg[5][1], obs[sg[6]]))
        ms_p = _time_ms(lambda: F.filter(eq_q, eq_r, m=M, e=E, n=n,
                                         fmt=binding.SS_FMT_SLICED2),
                        reps, F.sync)
        out.append({"E": E, "ms": ms, "pairs_per_s": n / (ms * 1e-3),
                    "hbm_gbs": gbs,
                    "hbm_frac": gbs / measured_peaks()["hbm_gbs"],
                    "accept_rate": float(acc.float().mean().item()),
                    "sliced_segments_ms": ms_s,
                    "sliced_segments_hbm_frac":
                        sliced_bytes / (ms_s * 1e-3) / 1e9
                        / measured_peaks()["hbm_gbs"],
                    "plain_sliced_equal_ms": ms_p,
                    "sliced_segments_over_plain_sliced": ms_s / ms_p})
    F.sync()
    return {"workload": f"{n // 1000000}M reads of {M} bp vs reference "
                        f"windows of {M - 8}..{M + 16} bp (flanked or cut)",
            "pairs": n, "per_E": out,
            "sliced_segments": f"{len(segs)} segments by window length, "
                               "one ss_filter_segments call per E",
            "results_identical": same}


def run_compaction(F, pq, pr, acc, n, E) -> dict:
    """The accepted pairs of one sweep launch compacted into an index list
    and gathered into dense packed buffers (the aligner's input)."""
    import torch

    from paper_1910_09020_gb300 import binding
    lib = binding.load()
    w16 = binding.ss_packed_words(M)
    idx = torch.empty(n, dtype=torch.int64, device=pq.device)
    cnt = torch.empty(1, dtype=torch.int64, device=pq.device)
    gq = torch.empty(n * w16, dtype=torch.int32, device=pq.device)
    gr = torch.empty_like(gq)
    st = torch.cuda.current_stream().cuda_stream

    def compact():
        binding._check(lib.ss_compact_accepted(
            F.ctx, acc.data_ptr(), n, st, idx.data_ptr(), cnt.data_ptr()),
            "ss_compact_accepted")

    def gather():
        binding._check(lib.ss_gather_pairs(
            F.ctx, pq.data_ptr(), pr.data_ptr(), M, idx.data_ptr(),
            cnt.data_ptr(), n, st, gq.data_ptr(), gr.data_ptr()),
            "ss_gather_pairs")

    compact()
    gather()
    torch.cuda.synchronize()
    c = int(cnt.item())
    out = {"E": E, "pairs": n, "accepted": c}
    for name, fn, nbytes in (
            ("compact", compact, 2 * n + 8 * c + 8),
            # per accepted pair: its index read, its words read and written
            ("gather", gather, c * (8 + 16 * w16))):
        a, b = _ev(), _ev()
        a.record()
        for _ in range(5):
            fn()
        b.record()
        torch.cuda.synchronize()
        ms = a.elapsed_time(b) / 5
        gbs = nbytes / (ms * 1e-3) / 1e9
        out[name] = {"ms": ms, "hbm_gbs": gbs,
                     "hbm_frac": gbs / measured_peaks()["hbm_gbs"]}
    F.sync()
    return out


def _pool_model(pool, ipk, sample=400, seed=1910_09020 + 55):
    """Op model of the served pool (the cheaper formulation per threshold
    group, as for the uneven batch) from the oracle's counters on `sample`
    pairs drawn uniformly from all of the pool's pairs: per-pair ALU and
    find-first ops, and the oracle's time on them."""
    counts = np.array([len(r[2]) for r in pool])
    owner = np.repeat(np.arange(len(pool)), counts)
    within = np.concatenate([np.arange(c) for c in counts])
    pick = np.sort(np.random.default_rng(seed).choice(
        len(owner), min(sample, len(owner)), replace=False))
    offs = [np.concatenate([[0], np.cumsum(r[2])]) for r in pool]
    L = np.array([pool[owner[i]][2][within[i]] for i in pick], np.int32)
    E = np.array([pool[owner[i]][3][within[i]] for i in pick], np.int32)
    rd = np.concatenate([pool[owner[i]][0][offs[owner[i]][within[i]]:
                                           offs[owner[i]][within[i] + 1]]
                         for i in pick])
    rf = np.concatenate([pool[owner[i]][1][offs[owner[i]][within[i]]:
                                           offs[owner[i]][within[i] + 1]]
                         for i in pick])
    off = np.concatenate([[0], np.cumsum(L.astype(np.int64))])
    t, alu, xu, _ = _oracle_model((rd, rf, off), L, E, np.arange(len(L)))
    return alu / len(L), xu / len(L), t, len(L)


def run_serving(seconds: float, slots: int = 2, ipk=None) -> dict:
    """Requests of 1..4096 pairs (log-uniform), lengths log-uniform
    100..100000 bp, edit rate U[0, 0.15], E = 10 % of length, arriving as a
    Poisson process at 30 %, 60 %, 75 % and 90 % of the measured (burst)
    capacity."""
    import queue
    import threading

    import torch

    from paper_1910_09020_gb300 import binding, synth
    pool = []
    for i in range(96):
        rng = np.random.default_rng(1910_09020 + 5 + i)
        n = int(np.exp(rng.uniform(0, np.log(4096))))
        L = synth.log_uniform(1910_09020 + 5000 + i, 0, n, 100, 100000)
        E = synth.thresholds(L, 10)
        reads, refs, _ = synth.pairs_varlen(1910_09020 + 50000 + i, 0, L,
                                            synth.rate_recipe(0.15))
        pinned = []
        for a in (reads, refs):  # pinned host memory copies fastest
            t = torch.empty(max(len(a), 1), dtype=torch.uint8,
                            pin_memory=True)
            t.numpy()[:len(a)] = a
            pinned.append(t.numpy()[:len(a)])
        pool.append((pinned[0], pinned[1], L, E))
    out = {"workload": "requests of 1..4096 pairs (log-uniform), lengths "
                       "log-uniform 100..100000 bp, edit rate U[0,0.15], "
                       "E = 10 % of length, Poisson arrivals",
           "slots": slots,
           "form": "host admission into slots; each batch's pass on its "
                   "slot, its CTA-per-pair pairs in the device-resident "
                   "ring drained by one long-lived worker kernel"}
    with binding.Server(0, hbm_budget_bytes=32 << 30, slots=slots) as S:
        # capacity: the whole pool at once, three times; the first warms
        # up and the faster of the other two counts (one burst's time moves
        # with the order its long pairs land in batches)
        dt = float("inf")
        for rep in range(3):
            S.reset_stats()
            t0 = time.perf_counter()
            ts = [S.submit(*r) for r in pool]
            for t in ts:
                S.wait(t)
            if rep > 0:
                dt = min(dt, time.perf_counter() - t0)
            for t in ts:
                S.fetch(t)
        pairs = sum(len(r[2]) for r in pool)
        cap_pairs = pairs / dt
        cap_req = len(pool) / dt
        out["capacity"] = {"pairs_per_s": cap_pairs, "requests_per_s": cap_req,
                           "gbases_per_s": sum(int(r[2].sum()) for r in pool)
                           / dt / 1e9}
        if ipk:
            # the burst's roofline: the pool's ALU work (op model) at the
            # LOP3 peak against the measured burst; the host link and HBM
            # bytes (2 m ASCII bytes per pair) are far below their rates
            alu, xu, t_o, k = _pool_model(pool, ipk)
            t_alu = alu * pairs / ipk["lop3"]
            t_xu = xu * pairs / ipk["bfind"]
            t = max(t_alu, t_xu)
            out["capacity"]["roofline"] = {
                "bound": "alu" if t == t_alu else "xu",
                "t_alu_s": t_alu, "t_xu_s": t_xu, "burst_s": dt,
                "alu_ops_per_pair": alu, "frac": t / dt,
                "model": "every row of the maze, of which the index "
                         "evaluates only a few: no bound of it",
                "sample": f"op model from the oracle on {k} pairs drawn "
                          f"uniformly from the pool ({t_o:.1f} s)"}
        loads = []
        for frac in (0.3, 0.6, 0.75, 0.9):
            rate = frac * cap_req
            nreq = max(20, int(rate * seconds))
            arr = synth.poisson_arrivals(1910_09020 + int(frac * 100), nreq,
                                         rate)
            pick = np.random.default_rng(int(frac * 1000)).integers(
                0, len(pool), nreq)
            S.reset_stats()
            # a client thread fetches each result as soon as it is done,
            # while requests keep arriving: a batch holds its device memory
            # (within the server's budget) until its results are fetched
            todo = queue.Queue()

            def fetcher():
                while True:
                    t = todo.get()
                    if t is None:
                        return
                    S.wait(t)
                    S.fetch(t)
            th = threading.Thread(target=fetcher)
            th.start()
            t0 = time.perf_counter()
            for k in range(nreq):
                delay = arr[k] - (time.perf_counter() - t0)
                if delay > 0:
                    time.sleep(delay)
                todo.put(S.submit(*pool[pick[k]]))
            todo.put(None)
            th.join()
            span = time.perf_counter() - t0
            st = S.stats()
            npairs = int(sum(len(pool[i][2]) for i in pick))
            loads.append({"offered_load": frac,
                          "offered_requests_per_s": rate,
                          "requests": nreq, "pairs": npairs,
                          "pairs_per_s": npairs / span,
                          "p50_s": st["latency_p50_s"],
                          "p99_s": st["latency_p99_s"],
                          "max_s": st["latency_max_s"],
                          "batches": st["batches"],
                          "max_inflight": st["max_inflight"],
                          "long_pairs_queued": st["long_pairs_queued"],
                          "worker_launches": st["worker_launches"]})
        out["loads"] = loads
    return out


# ---- our arm ---------------------------------------------------------------------

def run_ours(args):
    import torch

    from paper_1910_09020_gb300 import binding, synth
    from paper_1910_09020_gb300.peaks import measure as measure_int_peaks

    rank, world, local = dist_setup()
    n = args.pairs
    dev = torch.device("cuda", local)

    # inputs: generated into pinned host memory, copied once to HBM
    t0 = time.perf_counter()
    hq = torch.empty(n * M, dtype=torch.uint8, pin_memory=True)
    hr = torch.empty(n * M, dtype=torch.uint8, pin_memory=True)
    synth.pairs_fixed(SEED, rank * n, n, M, synth.SHORT_POISSON,
                      out=(hq.numpy(), hr.numpy()))
    gen_s = time.perf_counter() - t0
    dq = hq.to(dev, non_blocking=True)
    dr = hr.to(dev, non_blocking=True)
    torch.cuda.synchronize()

    F = binding.Filter(local, workspace_bytes=8 << 30)
    SL = binding.ss_sliced_words(M, n)
    sq = torch.empty(SL, dtype=torch.int32, device=dev)
    sr = torch.empty(SL, dtype=torch.int32, device=dev)
    acc = torch.empty((len(SWEEP), n), dtype=torch.uint8, device=dev)
    obs = torch.empty((len(SWEEP), n), dtype=torch.int32, device=dev)
    # events on the stream the library is called on (torch's current
    # stream; the sweep's launches on the library's other streams are
    # joined back into it before the call returns), one set per timed step
    evs = [[torch.cuda.Event(enable_timing=True) for _ in range(3)]
           for _ in range(args.steps)]
    launch_ms = {"pack": [], "filter": []}
    row = {E: t for t, E in enumerate(SWEEP)}

    def step(ev):
        if ev:
            ev[0].record()
        F.pack_sliced(dq, m=M, n=n, out=sq)
        F.pack_sliced(dr, m=M, n=n, out=sr)
        if ev:
            ev[1].record()
        F.filter_sweep(sq, sr, m=M, e=SWEEP, n=n, out_accept=acc,
                       out_obstacles=obs)
        if ev:
            ev[2].record()

    for _ in range(args.warmup):
        step(None)
    F.sync()
    torch.cuda.synchronize()

    clocks = ClockSampler(local)
    clocks.start()
    barrier(world)
    torch.cuda.synchronize()
    start, stop = (torch.cuda.Event(enable_timing=True),
                   torch.cuda.Event(enable_timing=True))
    start.record()
    for s in range(args.steps):
        step(evs[s])
    stop.record()
    torch.cuda.synchronize()
    for ev in evs:
        launch_ms["pack"].append(ev[0].elapsed_time(ev[1]))
        launch_ms["filter"].append(ev[1].elapsed_time(ev[2]))
    barrier(world)
    clk = clocks.stop()
    elapsed_ms = start.elapsed_time(stop)
    F.sync()
    elapsed_ms = max_over_ranks(elapsed_ms, world)
    pairs_per_step = n * len(SWEEP)
    value = world * pairs_per_step * args.steps / (elapsed_ms * 1e-3)

    # e2e: the public host-buffer call, copies inside the timed region
    e2e = None
    if not args.no_e2e:
        hacc = torch.empty((len(SWEEP), n), dtype=torch.uint8, pin_memory=True)
        hobs = torch.empty((len(SWEEP), n), dtype=torch.int32, pin_memory=True)
        hq2, hr2 = hq.view(n, M), hr.view(n, M)
        F.filter_host(hq2, hr2, m=M, e=SWEEP, fmt=binding.SS_FMT_ASCII,
                      out_accept=hacc, out_obstacles=hobs)
        # each step timed on its own; the value is taken from the median
        # step (a host-side transient, e.g. memory a previous process is
        # still releasing, slows single steps), the mean is reported beside
        e2e_steps = max(5, args.steps // 4)
        barrier(world)
        per_step = []
        for _ in range(e2e_steps):
            t0 = time.perf_counter()
            F.filter_host(hq2, hr2, m=M, e=SWEEP, fmt=binding.SS_FMT_ASCII,
                          out_accept=hacc, out_obstacles=hobs)
            per_step.append(time.perf_counter() - t0)
        dt = max_over_ranks(float(np.median(per_step)), world)
        dt_mean = max_over_ranks(float(np.mean(per_step)), world)
        e2e = {"value": world * pairs_per_step / dt,
               "unit": "pairs/s", "h2d_bytes_per_step": 2 * n * M,
               "d2h_bytes_per_step": 5 * n * len(SWEEP),
               "ms_per_step": 1e3 * dt, "steps": e2e_steps,
               "ms_per_step_mean": 1e3 * dt_mean,
               "ms_per_step_each": [1e3 * x for x in per_step]}
        # the device path and the host path must agree
        same = (torch.equal(hacc, acc.cpu()) and torch.equal(hobs, obs.cpu()))
        e2e["matches_device_path"] = bool(same)
        # the host link's own rate: pinned host -> device copies of the
        # same input bytes, the best of three (the e2e path cannot beat
        # bytes / this rate)
        best_ms = float("inf")
        for _ in range(3):
            a, b = _ev(), _ev()
            torch.cuda.synchronize()
            a.record()
            dq.copy_(hq, non_blocking=True)
            dr.copy_(hr, non_blocking=True)
            b.record()
            torch.cuda.synchronize()
            best_ms = min(best_ms, a.elapsed_time(b))
        h2d_gbs = 2 * n * M / (best_ms * 1e-3) / 1e9
        e2e["h2d_copy_gbs"] = h2d_gbs
        e2e["copy_bound_pairs_per_s"] = (
            world * pairs_per_step / (2 * n * M / (h2d_gbs * 1e9)))

    if rank != 0:
        F.close()
        import torch.distributed as dist
        dist.destroy_process_group()
        return 0

    # the same step in the pair-major packed format (one pair per thread),
    # beside the headline; its results must equal the sliced form's
    W16 = binding.ss_packed_words(M)
    pq = torch.empty(n * W16, dtype=torch.int32, device=dev)
    pr = torch.empty(n * W16, dtype=torch.int32, device=dev)
    pm_acc = torch.empty(n, dtype=torch.uint8, device=dev)
    pm_obs = torch.empty(n, dtype=torch.int32, device=dev)
    pair_major = {"per_E_ms": {}, "results_identical": True}
    pair_major["pack_ms"] = _time_ms(
        lambda: (F.pack(dq, m=M, n=n, out=pq), F.pack(dr, m=M, n=n, out=pr)),
        3, F.sync)
    for t, E in enumerate(SWEEP):
        pair_major["per_E_ms"][E] = _time_ms(
            lambda: F.filter(pq, pr, m=M, e=E, n=n, out_accept=pm_acc,
                             out_obstacles=pm_obs), 3, F.sync)
        pair_major["results_identical"] &= bool(
            torch.equal(pm_acc, acc[t]) and torch.equal(pm_obs, obs[t]))
    pair_major["step_ms"] = (pair_major["pack_ms"]
                             + sum(pair_major["per_E_ms"].values()))
    pair_major["pairs_per_s"] = (n * len(SWEEP)
                                 / (pair_major["step_ms"] * 1e-3))
    pair_major["kernels"] = "k_pack_fixed x2, k_rw_uniform<E> x6"

    # roofline of the dominant kernel: the filter launches of the sweep
    peaks = measured_peaks()
    ipk = measure_int_peaks(local)
    cpu = None
    model = None
    parity = None
    if not args.no_cpu and world == 1:
        cpu, stats, parity = cpu_oracle_full(
            hq.numpy().reshape(n, M), hr.numpy().reshape(n, M),
            acc.cpu().numpy(), obs.cpu().numpy())
        model = op_model(stats, n, M)
    hbm = peaks["hbm_gbs"] * 1e9
    # each launch of the sweep alone (outside the timed region, one after
    # the other on one stream), for the per-launch rooflines
    solo_ms = {}
    for grp in GROUPS:
        a0 = row[grp[0]]
        if len(grp) > 1:
            fn = (lambda grp=grp, a0=a0: F.filter_sweep(
                sq, sr, m=M, e=list(grp), n=n,
                out_accept=acc[a0:a0 + len(grp)],
                out_obstacles=obs[a0:a0 + len(grp)]))
        else:
            fn = (lambda grp=grp, a0=a0: F.filter(
                sq, sr, m=M, e=grp[0], n=n, fmt=binding.SS_FMT_SLICED2,
                out_accept=acc[a0], out_obstacles=obs[a0]))
        solo_ms[grp] = _time_ms(fn, 5, F.sync)
    per_launch = []
    roof_total = meas_total = 0.0
    sum_t = {"hbm": 0.0, "alu": 0.0, "xu": 0.0}
    for grp in GROUPS:
        ms = solo_ms[grp]
        # the pairs read once, each threshold's results written
        gbytes = FILTER_BYTES_PER_PAIR + 5 * (len(grp) - 1)
        t_hbm = n * gbytes / hbm
        sum_t["hbm"] += 1e3 * t_hbm
        d = {"E": grp[0] if len(grp) == 1 else list(grp), "ms": ms,
             "kernel": "k_sliced" if len(grp) == 1 else "k_sliced_set",
             "pairs_per_s": n / (ms * 1e-3),
             "hbm_gbs": n * gbytes / (ms * 1e-3) / 1e9,
             "algorithmic_bytes_per_pair": gbytes,
             "t_hbm_ms": 1e3 * t_hbm}
        t_bound, bound = t_hbm, "hbm"
        if model:
            alu = sum(model[E]["alu_ops_per_pair"] for E in grp)
            xu = sum(model[E]["xu_ops_per_pair"] for E in grp)
            t_alu = n * alu / ipk["lop3"]
            t_xu = n * xu / ipk["bfind"]
            sum_t["alu"] += 1e3 * t_alu
            sum_t["xu"] += 1e3 * t_xu
            d.update({"t_alu_ms": 1e3 * t_alu, "t_xu_ms": 1e3 * t_xu,
                      "model": [model[E]["model"] for E in grp],
                      "alu_ops_per_pair": alu,
                      "alu_ops_row_words_per_pair": sum(
                          model[E]["alu_ops_row_words_per_pair"]
                          for E in grp),
                      "alu_ops_columns_per_pair": sum(
                          model[E]["alu_ops_columns_per_pair"] for E in grp),
                      "alu_ops_sliced_per_pair": sum(
                          model[E].get("alu_ops_sliced_per_pair", 0)
                          for E in grp),
                      "columns_per_pair": [model[E]["columns_per_pair"]
                                           for E in grp],
                      "tops": n * alu / (ms * 1e-3) / 1e12})
            if len(grp) == 1:
                d["model"] = d["model"][0]
                d["columns_per_pair"] = d["columns_per_pair"][0]
            if max(t_alu, t_xu) > t_bound:
                t_bound, bound = max(t_alu, t_xu), ("alu" if t_alu >= t_xu
                                                    else "xu")
        d["bound"] = bound
        d["frac"] = 1e3 * t_bound / ms
        roof_total += 1e3 * t_bound
        meas_total += ms
        per_launch.append(d)
    # the step's filter section (the sweep call, launches side by side),
    # timed in the timed region; its roofline time is the largest of the
    # summed HBM, logic-pipe and find-first times of its launches (they
    # share the GPU's bandwidth and pipes)
    filter_ms = float(np.mean(launch_ms["filter"]))
    pack_ms = float(np.mean(launch_ms["pack"]))
    dom_bound = max(sum_t, key=sum_t.get)
    if dom_bound == "hbm":
        achieved = sum(n * d["algorithmic_bytes_per_pair"]
                       for d in per_launch) / (filter_ms * 1e-3) / 1e9
        peak, unit = peaks["hbm_gbs"], "GB/s"
    elif dom_bound == "alu":
        ops = sum(n * model[E]["alu_ops_per_pair"] for E in SWEEP)
        achieved = ops / (filter_ms * 1e-3) / 1e12
        peak, unit = ipk["lop3"] / 1e12, "Tops/s"
    else:
        ops = sum(n * model[E]["xu_ops_per_pair"] for E in SWEEP)
        achieved = ops / (filter_ms * 1e-3) / 1e12
        peak, unit = ipk["bfind"] / 1e12, "Tops/s"
    # DRAM bytes of the section: each launch's ncu figure per pair
    per_kernel = [ncu_traffic("k_sliced" if len(grp) == 1 else
                              "k_sliced_set") for grp in GROUPS]
    traffic = (None if any(t is None for t in per_kernel)
               else n * sum(per_kernel))
    roofline = {
        "kernel": "k_sliced / k_sliced_set (plain filter over the "
                  "bit-sliced layout: E = 0, 2, 4 in one shared pass, "
                  "E = 6, 8, 10 one launch each, side by side)",
        "bound": dom_bound, "achieved": achieved, "peak": peak, "unit": unit,
        "frac": max(sum_t.values()) / filter_ms,
        "filter_section_ms": filter_ms,
        "t_section_ms": sum_t,
        "frac_launches_alone": roof_total / meas_total,
        "frac_note": "the step's filter section (one ss_filter_sweep call, "
                     "its 4 launches side by side, timed by events in the "
                     "timed region): max over HBM, ALU and find-first of "
                     "the launches' summed roofline times / the section's "
                     "time.  frac_launches_alone: the sum over the launches "
                     "of max(HBM, ALU, find-first) / the sum of their times "
                     "each launched alone (per_launch; a shared "
                     "pass: the pairs read once, each threshold's results "
                     "written, the ALU ops of all its thresholds); the ALU "
                     "term counts "
                     "the cheapest of three formulations of the greedy for "
                     "each E (per_launch[].model): row words, columns one "
                     "pair per thread, bit-sliced columns (32 pairs per "
                     "word, every column walked)",
        "traffic": traffic,
        "algorithmic_bytes_per_launch": n * FILTER_BYTES_PER_PAIR,
        "algorithmic_bytes_section": sum(n * d["algorithmic_bytes_per_pair"]
                                         for d in per_launch),
        "peak_source": f"HBM {peaks['hbm_source']} ({peaks['hbm_gbs']} GB/s); "
                       "integer pipes measured live by microbenchmark",
        "int_peaks_tops": {k: v / 1e12 for k, v in ipk.items()},
        "per_launch": per_launch,
    }
    # accuracy of the decisions just timed (Section 3.2's rates), against the
    # banded edit-distance verifier; outside the timed region
    accuracy = []
    for t, E in enumerate(SWEEP):
        ed = F.edit_distance(pq, pr, m=M, e=E, n=n)
        ev_a, ev_b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(
            enable_timing=True)
        ev_a.record()
        F.edit_distance(pq, pr, m=M, e=E, n=n, out=ed)
        ev_b.record()
        ta, fa, fr, tr = F.confusion(acc[t], ed, e=E)
        accuracy.append({"E": E, "true_accepts": ta, "false_accepts": fa,
                         "false_rejects": fr, "true_rejects": tr,
                         "false_accept_rate": fa / max(fa + tr, 1),
                         "false_reject_rate": fr / max(fr + ta, 1),
                         "verifier_ms": ev_a.elapsed_time(ev_b)})
    F.sync()

    extras = {}
    if not args.headline_only and world == 1:
        extras["submaze_t8_y3"] = run_submaze(F, sq, sr, pq, pr, n, acc,
                                              obs)
        extras["unequal_lengths"] = run_unequal(F)
        k4 = SWEEP.index(4)
        extras["compaction"] = run_compaction(F, pq, pr, acc[k4], n, 4)
        del dq, dr, pq, pr, sq, sr
        torch.cuda.empty_cache()
        extras["persistent_uneven_batch"] = run_batched(
            F, ipk, peaks["hbm_gbs"], not args.no_cpu,
            n=args.batched_pairs)
        torch.cuda.empty_cache()
        extras["plain_vs_persistent_two_lengths"] = run_two_lengths(
            F, ipk, peaks["hbm_gbs"])
        torch.cuda.empty_cache()
        extras["served"] = run_serving(args.serve_seconds, ipk=ipk)
    line = {
        "metric": METRIC, "value": value, "unit": "pairs/s",
        "gbases_per_s": value * M / 1e9, "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": elapsed_ms / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "u32",
        "data": "synthetic", "config": config_dict(world, n),
        "clocks": clk, "e2e": e2e,
        "gpu_launches": (2 + len(GROUPS)) * args.steps,
        "roofline": roofline, "cpu_baseline": cpu, "parity": parity,
        "breakdown": {"pack_ms": pack_ms, "filter_ms": filter_ms,
                      "pack_gbs": n * PACK_BYTES_PER_PAIR / (pack_ms * 1e-3)
                      / 1e9, "generate_s": gen_s},
        "pair_major_form": pair_major,
        "accuracy": accuracy,
        **extras,
    }
    print_line(line, args.details)
    F.close()
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()
    return 0


def run_batched_only(args):
    """The persistent launch of the uneven batch alone (profiling aid)."""
    import torch

    from paper_1910_09020_gb300 import binding
    torch.cuda.set_device(0)
    F = binding.Filter(0, workspace_bytes=8 << 30)
    out = run_batched(F, None, measured_peaks()["hbm_gbs"], False,
                      per_length_too=False, n=args.batched_pairs)
    print(json.dumps(out), flush=True)
    F.close()
    return 0


def run_two_lengths_only(args):
    """The two-length comparison of forms alone (10M x 250 bp + 10M x 150
    bp, E = 0..10 % of length)."""
    import torch

    from paper_1910_09020_gb300 import binding
    from paper_1910_09020_gb300.peaks import measure as measure_int_peaks
    torch.cuda.set_device(0)
    F = binding.Filter(0, workspace_bytes=8 << 30)
    out = run_two_lengths(F, measure_int_peaks(0), measured_peaks()["hbm_gbs"])
    print(json.dumps(out), flush=True)
    F.close()
    return 0


def run_long_only(args):
    """One index class alone (profiling aid): 608 pairs of 20 kbp, edit rate
    5 %, E = 10 % of the length (2000), the shape of the served form's long
    pairs.  Two filter passes without graph replay, so that a profiler sees
    every launch; the busy launches are those of k_cw_index<1>."""
    import torch

    from paper_1910_09020_gb300 import binding, synth
    torch.cuda.set_device(0)
    F = binding.Filter(0, workspace_bytes=1 << 30)
    F.set_tuning(31, 8)
    n, m = 608, 20000
    L = np.full(n, m, np.int32)
    E = synth.thresholds(L, 10)
    pq, pr, dwo, dL, _, _ = _pack_varlen(F, L, synth.rate_recipe(0.05), 5)
    dE = torch.from_numpy(E).cuda()
    times = []
    for _ in range(2):
        t0 = time.perf_counter()
        acc, obs = F.filter(pq, pr, offsets=dwo, lengths=dL, E=dE, sync=True,
                            flags=binding.SS_FLAG_NO_GRAPH)
        times.append(time.perf_counter() - t0)
    o = obs.cpu().numpy()
    print(json.dumps({"workload": f"{n} pairs x {m} bp, E = {int(E[0])}, "
                                  "edit rate 5 %, k_cw_index<1>",
                      "ms": [round(1e3 * t, 3) for t in times],
                      "greedy_iterations": int(o.sum()),
                      "accepted": int(acc.sum().item())}), flush=True)
    F.close()
    return 0


def main():
    args = parse()
    if args.impl == "reference":
        return run_reference(args)
    if args.workload == "batched":
        return run_batched_only(args)
    if args.workload == "two_lengths":
        return run_two_lengths_only(args)
    if args.workload == "long":
        return run_long_only(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
