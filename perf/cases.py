"""Workloads the library is timed on: what a user of the filter has it do,
through the public entry points of ``paper_1910_09020_gb300.binding``.

Every case is one kind of call at one size.  ``listed()`` names the sizes the
configurations, tests and benchmark of this repository use; ``draw()`` gives
more of the same kinds over the whole range of lengths, thresholds and pair
counts.  Inputs are random reads and references made on the GPU from a seed:
a reference is the read with substitutions, insertions and deletions at a
rate of its own, cut or padded with random bases.
"""
import math

import numpy as np
import torch

from paper_1910_09020_gb300 import binding

# substitutions, insertions, deletions
EVEN_MIX = (1 / 3, 1 / 3, 1 / 3)
READ_MIX = (0.8, 0.1, 0.1)


def listed():
    return [
        # one small batch of ASCII pairs already on the GPU, as a mapper's
        # first stage hands over: latency and launches count
        {"name": "small_batch", "kind": "batch", "n": 10_000, "m": 100,
         "e": 5},
        # 30M short pairs packed once and filtered at six thresholds: the
        # threshold sweep of the benchmark, half of the pairs unrelated
        {"name": "sweep_30M", "kind": "sweep", "n": 30_000_000, "m": 100},
        # a batch of two read lengths, already in the bit-sliced layout, each
        # length at 5 % of it
        {"name": "two_lengths", "kind": "segments", "n1": 4_000_000,
         "m1": 250, "n2": 4_000_000, "m2": 150, "percent": 5},
        # a mapper's pipeline in the default (pair-major) format: pack,
        # filter, list the accepted pairs and gather them for an aligner
        {"name": "mapper_150bp", "kind": "mapper", "n": 4_000_000, "m": 150,
         "e": 7},
        # lengths and thresholds of their own per pair, 64 bp to 10 kbp
        {"name": "uneven_2M", "kind": "uneven", "n": 2_000_000, "lo": 64,
         "hi": 10_000, "percent": 5, "rmax": 0.10},
        # long reads: 10 to 100 kbp at 10 % of the length
        {"name": "long_reads", "kind": "uneven", "n": 1_000, "lo": 10_000,
         "hi": 100_000, "percent": 10, "rmax": 0.15},
        # the server given a burst of requests of 1 to 4096 pairs of 100 bp
        # to 100 kbp, each result fetched as it completes
        {"name": "served_burst", "kind": "served", "requests": 24,
         "pairs": 4096, "lo": 100, "hi": 100_000},
        # a sweep over pairs held in pinned host memory
        {"name": "host_stream", "kind": "host", "n": 4_000_000, "m": 100},
        # reads against candidate windows of lengths of their own
        {"name": "windows_2M", "kind": "unequal", "n": 2_000_000, "m": 100,
         "below": 8, "above": 16, "e": 6},
        # the sub-maze approximate mode at the paper's t = 8, y = 3
        {"name": "submaze_4M", "kind": "submaze", "n": 4_000_000, "m": 100,
         "e": 5, "t": 8, "y": 3},
        # exact capped distances of short pairs, the accuracy harness'
        # ground truth for the filter's decisions
        {"name": "distance_100bp", "kind": "distance", "n": 3_000_000,
         "m": 100, "e": 5},
        # the same for pairs of lengths and thresholds of their own
        {"name": "distance_uneven", "kind": "distance_uneven", "n": 60_000,
         "lo": 64, "hi": 10_000, "percent": 5, "rmax": 0.10},
    ]


def _log(rng, lo, hi):
    """An integer of lo..hi, uniform in its logarithm."""
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo),
                                                    math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["batch", "sweep", "segments", "mapper", "uneven",
                       "long", "served", "host", "unequal", "submaze",
                       "distance", "distance_uneven"])
    m = _log(rng, 64, 300)
    if kind == "batch":
        return {"kind": kind, "n": _log(rng, 1_000, 3_000_000), "m": m,
                "e": rng.randint(0, min(31, m // 10))}
    if kind == "sweep":
        return {"kind": kind, "m": m,
                "n": min(_log(rng, 200_000, 30_000_000), 3_000_000_000 // m)}
    if kind == "segments":
        return {"kind": kind, "n1": _log(rng, 20_000, 4_000_000),
                "m1": _log(rng, 64, 250), "n2": _log(rng, 20_000, 4_000_000),
                "m2": _log(rng, 64, 250), "percent": rng.randint(0, 10)}
    if kind == "mapper":
        return {"kind": kind, "n": _log(rng, 20_000, 600_000_000 // m),
                "m": m, "e": rng.randint(1, min(31, m // 10))}
    if kind == "uneven":
        percent = rng.randint(1, 10)
        return {"kind": kind, "lo": 64, "hi": _log(rng, 500, 10_000),
                "n": _log(rng, 20_000, 2_000_000 * 5 // max(percent, 5)),
                "percent": percent, "rmax": 0.10}
    if kind == "long":
        return {"kind": "uneven", "lo": 10_000,
                "hi": _log(rng, 20_000, 100_000), "n": _log(rng, 50, 1_000),
                "percent": rng.randint(1, 10), "rmax": 0.15}
    if kind == "served":
        return {"kind": kind, "requests": rng.randint(4, 24),
                "pairs": _log(rng, 64, 4096), "lo": 100,
                "hi": _log(rng, 2_000, 100_000)}
    if kind == "host":
        return {"kind": kind, "m": m,
                "n": _log(rng, 50_000, 400_000_000 // m)}
    if kind == "unequal":
        return {"kind": kind, "n": _log(rng, 20_000, 200_000_000 // m),
                "m": m, "below": rng.randint(0, 16),
                "above": rng.randint(0, 32),
                "e": rng.randint(1, min(15, m // 10))}
    if kind == "submaze":
        return {"kind": kind, "n": _log(rng, 20_000, 400_000_000 // m),
                "m": m, "e": rng.randint(1, min(31, m // 10)),
                "t": rng.randint(4, 16), "y": rng.randint(1, 4)}
    if kind == "distance":
        return {"kind": kind, "n": _log(rng, 20_000, 300_000_000 // m),
                "m": m, "e": rng.randint(1, min(10, m // 10))}
    percent = rng.randint(1, 5)
    return {"kind": "distance_uneven", "lo": 64,
            "hi": _log(rng, 500, 10_000), "n": _log(rng, 2_000, 60_000),
            "percent": percent, "rmax": 0.10}


# ---- inputs ---------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _codes(g, n):
    return torch.randint(0, 4, (n,), dtype=torch.uint8, device="cuda",
                         generator=g)


def _ascii(codes):
    letters = torch.tensor([65, 67, 71, 84], dtype=torch.uint8, device="cuda")
    return letters[codes.to(torch.int32)]


def _pairs(g, lengths, rate, mix, unrelated=None):
    """Concatenated ASCII reads and references of the given lengths (int64,
    CUDA): each reference base is edited with its pair's rate; the pairs of
    the mask `unrelated` get a random reference."""
    off = torch.cumsum(lengths, 0)
    total = int(off[-1])
    reads = torch.empty(total, dtype=torch.uint8, device="cuda")
    refs = torch.empty_like(reads)
    ends = off.cpu().numpy()
    psub, pins = mix[0], mix[0] + mix[1]
    a, first = 0, 0
    while a < len(ends):
        b = max(a + 1, int(np.searchsorted(ends, first + (1 << 26), "right")))
        last = int(ends[b - 1])
        size = last - first
        part = lengths[a:b]
        pid = torch.repeat_interleave(
            torch.arange(b - a, device="cuda", dtype=torch.int32), part,
            output_size=size)
        end = off[a:b] - first
        begin = end - part
        read = _codes(g, size)
        other = _codes(g, size)
        u = torch.rand(size, device="cuda", generator=g) / rate[a:b][pid]
        ins = (u >= psub) & (u < pins)
        gone = (u >= pins) & (u < 1.0)
        run = torch.cumsum(gone.to(torch.int8) - ins.to(torch.int8), 0,
                           dtype=torch.int32)
        before = torch.where(begin > 0, run[(begin - 1).clamp(min=0)], 0)
        src = torch.arange(size, device="cuda", dtype=torch.int32)
        src += run + ins.to(torch.int32) - before[pid]
        keep = (src < end.to(torch.int32)[pid]) & ~ins
        ref = torch.where(keep, read[src.clamp(0, size - 1)], other)
        ref = torch.where(u < psub, (ref + 1 + other % 3) & 3, ref)
        if unrelated is not None:
            ref = torch.where(unrelated[a:b][pid], other, ref)
        reads[first:last] = _ascii(read)
        refs[first:last] = _ascii(ref)
        a, first = b, last
    return reads, refs


def _fixed(g, n, m, rate, mix, unrelated=None):
    lengths = torch.full((n,), m, dtype=torch.int64, device="cuda")
    return _pairs(g, lengths, rate, mix, unrelated)


def _short(g, n, m):
    """Pairs like the benchmark's: even ones with a few edits (three per 100
    bases), odd ones unrelated."""
    rate = torch.full((n,), 0.03, device="cuda")
    odd = torch.arange(n, device="cuda") % 2 == 1
    return _fixed(g, n, m, rate, EVEN_MIX, odd)


def _rates(g, n, top):
    return torch.rand(n, device="cuda", generator=g) * top + 1e-6


def _log_lengths(g, n, lo, hi):
    """Lengths log-uniform in lo..hi, one from each of n equal parts of the
    range in random order, so that every seed has the same work."""
    u = (torch.randperm(n, device="cuda", generator=g).double()
         + torch.rand(n, device="cuda", generator=g).double()) / n
    x = torch.exp(math.log(lo) + u * (math.log(hi + 1) - math.log(lo)))
    return x.to(torch.int64).clamp(lo, hi)


def _uneven(F, case, seed):
    """Pairs of lengths of their own, packed: the filter's and the
    verifier's mixed input."""
    g = _gen(seed)
    n = case["n"]
    length = _log_lengths(g, n, case["lo"], case["hi"])
    reads, refs = _pairs(g, length, _rates(g, n, case["rmax"]), READ_MIX)
    words = (length + 15) // 16
    woff = torch.cumsum(words, 0) - words
    boff = torch.cumsum(length, 0) - length
    short = length.to(torch.int32)
    packed = []
    for side in (reads, refs):
        out = torch.empty(int(words.sum()), dtype=torch.int32, device="cuda")
        packed.append(F.pack(side, offsets=boff, lengths=short, out=out,
                             out_offsets=woff))
    return {"q": packed[0], "r": packed[1], "off": woff, "len": short,
            "E": (length * case["percent"] // 100).to(torch.int32)}


def _percent(m, percent):
    return min(31, m * percent // 100)


def _sweep(m):
    """The benchmark's thresholds, 0 to 10 % of the length."""
    return [_percent(m, p) for p in (0, 2, 4, 6, 8, 10)]


def _windows(case, seed):
    """Reads of m bases and windows of m - below .. m + above bases: the
    edited read between random flanks, or cut."""
    g = _gen(seed)
    n, m = case["n"], case["m"]
    reads, core = _fixed(g, n, m, _rates(g, n, 0.12), READ_MIX)
    d = torch.randint(-case["below"], case["above"] + 1, (n,), device="cuda",
                      generator=g)
    flank = (torch.rand(n, device="cuda", generator=g)
             * (d.clamp(min=0) + 1)).long()
    length = m + d
    off = torch.cumsum(length, 0) - length
    pid = torch.repeat_interleave(torch.arange(n, device="cuda"), length)
    col = torch.arange(pid.numel(), device="cuda") - off[pid] - flank[pid]
    inside = (col >= 0) & (col < m)
    refs = torch.where(inside, core[pid * m + col.clamp(0, m - 1)],
                       _ascii(_codes(g, pid.numel())))
    return reads, refs, length, off


def prepare(case, seed):
    kind = case["kind"]
    g = _gen(seed)
    if kind == "served":
        return _prepare_served(case, seed)
    F = binding.Filter(0)
    s = {"case": case, "F": F}
    if kind in ("uneven", "distance_uneven"):
        s.update(_uneven(F, case, seed))
    elif kind == "batch":
        n, m = case["n"], case["m"]
        edits = torch.randint(0, 11, (n,), device="cuda", generator=g)
        s["q"], s["r"] = _fixed(g, n, m, edits / 100 + 1e-6, EVEN_MIX)
    elif kind in ("sweep", "host"):
        s["q"], s["r"] = _short(g, case["n"], case["m"])
        if kind == "host":
            shape = (6, case["n"])
            for k in ("q", "r"):
                host = torch.empty(s[k].shape, dtype=torch.uint8,
                                   pin_memory=True)
                s[k] = host.copy_(s[k])
            s["acc"] = torch.empty(shape, dtype=torch.uint8, pin_memory=True)
            s["obs"] = torch.empty(shape, dtype=torch.int32, pin_memory=True)
    elif kind == "segments":
        s["seg"] = []
        for n, m in ((case["n1"], case["m1"]), (case["n2"], case["m2"])):
            q, r = _fixed(g, n, m, _rates(g, n, 0.12), READ_MIX)
            s["seg"].append((F.pack_sliced(q, m=m, n=n),
                             F.pack_sliced(r, m=m, n=n), m,
                             _percent(m, case["percent"]), n))
    elif kind == "mapper":
        n, m = case["n"], case["m"]
        s["q"], s["r"] = _fixed(g, n, m, _rates(g, n, 0.12), READ_MIX)
    elif kind == "unequal":
        reads, refs, length, off = _windows(case, seed)
        n, m = case["n"], case["m"]
        s["q"] = F.pack(reads, m=m, n=n)
        s["qoff"] = (torch.arange(n, device="cuda")
                     * binding.ss_packed_words(m))
        s["qlen"] = torch.full((n,), m, dtype=torch.int32, device="cuda")
        words = (length + 15) // 16
        s["roff"] = torch.cumsum(words, 0) - words
        s["rlen"] = length.to(torch.int32)
        out = torch.empty(int(words.sum()), dtype=torch.int32, device="cuda")
        s["r"] = F.pack(refs, offsets=off, lengths=s["rlen"], out=out,
                        out_offsets=s["roff"])
    else:  # submaze, distance: fixed-length pairs in the packed format
        n, m = case["n"], case["m"]
        q, r = _short(g, n, m)
        s["q"], s["r"] = F.pack(q, m=m, n=n), F.pack(r, m=m, n=n)
    F.sync()
    return s


def _request_sizes(case):
    """Pairs per request, log-uniform in 1..pairs (the same for any seed)."""
    k = case["requests"]
    return [int(math.exp((i + 0.5) / k * math.log(case["pairs"])))
            for i in range(k)]


def _prepare_served(case, seed):
    """Requests in pinned host memory, in random order of size."""
    sizes = _request_sizes(case)
    order = np.random.default_rng(int(seed)).permutation(len(sizes))
    g = _gen(seed)
    total = sum(sizes)
    length = _log_lengths(g, total, case["lo"], case["hi"])
    sides = []
    for side in _pairs(g, length, _rates(g, total, 0.15), READ_MIX):
        host = torch.empty(side.shape, dtype=torch.uint8, pin_memory=True)
        sides.append(host.copy_(side))
    L = length.to(torch.int32).cpu().numpy()
    E = (length * 10 // 100).to(torch.int32).cpu().numpy()
    byte = np.concatenate([[0], np.cumsum(L, dtype=np.int64)])
    requests, a = [], 0
    for i in order:
        b = a + sizes[i]
        requests.append(tuple(x.numpy()[byte[a]:byte[b]] for x in sides)
                        + (L[a:b], E[a:b]))
        a = b
    return {"case": case, "S": binding.Server(0, hbm_budget_bytes=32 << 30,
                                              slots=2),
            "requests": requests}


# ---- one pass ----------------------------------------------------------------

def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "served":
        S = s["S"]
        tickets = [S.submit(*r) for r in s["requests"]]
        acc, obs = [], []
        for t in tickets:
            S.wait(t)
            _, a, o, _ = S.fetch(t)
            acc.append(a)
            obs.append(o)
        return np.concatenate(acc), np.concatenate(obs)
    F = s["F"]
    if kind in ("uneven", "distance_uneven"):
        if kind == "uneven":
            return F.filter(s["q"], s["r"], offsets=s["off"],
                            lengths=s["len"], E=s["E"])
        return F.edit_distance_varlen(s["q"], s["r"], s["off"], s["len"],
                                      s["E"])
    if kind == "segments":
        return F.filter_segments(s["seg"])
    if kind == "unequal":
        return F.filter_unequal(s["q"], s["qoff"], s["qlen"], s["r"],
                                s["roff"], s["rlen"], e=case["e"])
    n, m = case["n"], case["m"]
    if kind == "batch":
        return F.filter(s["q"], s["r"], m=m, e=case["e"], n=n,
                        fmt=binding.SS_FMT_ASCII)
    if kind == "sweep":
        q = F.pack_sliced(s["q"], m=m, n=n)
        r = F.pack_sliced(s["r"], m=m, n=n)
        return F.filter_sweep(q, r, m=m, e=_sweep(m), n=n)
    if kind == "host":
        return F.filter_host(s["q"], s["r"], m=m, e=_sweep(m), n=n,
                             out_accept=s["acc"], out_obstacles=s["obs"])
    if kind == "mapper":
        q = F.pack(s["q"], m=m, n=n)
        r = F.pack(s["r"], m=m, n=n)
        acc, obs = F.filter(q, r, m=m, e=case["e"], n=n)
        # the index list is defined up to count only: the gathered pairs
        # (zero past count) show it whole
        index, count = F.compact(acc)
        gq, gr = F.gather(q, r, index, count, m=m, n=n)
        return acc, obs, count, gq, gr
    if kind == "submaze":
        return F.filter_submaze(s["q"], s["r"], m=m, e=case["e"],
                                t=case["t"], y=case["y"], n=n)
    return F.edit_distance(s["q"], s["r"], m=m, e=case["e"], n=n)


# ---- what one pass cannot do without -------------------------------------------

def _mean_log(lo, hi):
    return (hi - lo) / math.log(hi / lo) if hi > lo else lo


def work(case):
    """Bytes: every input read once, every output written once.  Operations:
    one comparison per reference base, pair and threshold."""
    kind = case["kind"]
    if kind == "served":
        n = sum(_request_sizes(case))
        bases = n * _mean_log(case["lo"], case["hi"])
        return {"bytes": 2 * bases + 13 * n, "flops": bases}
    if kind in ("uneven", "distance_uneven"):
        n = case["n"]
        bases = n * _mean_log(case["lo"], case["hi"])
        out = 5 if kind == "uneven" else 4
        return {"bytes": bases / 2 + (16 + out) * n, "flops": bases}
    if kind == "segments":
        sizes = ((case["n1"], case["m1"]), (case["n2"], case["m2"]))
        return {"bytes": sum(n * (m / 2 + 5) for n, m in sizes),
                "flops": sum(n * m for n, m in sizes)}
    n, m = case["n"], case["m"]
    if kind == "batch":
        return {"bytes": n * (2 * m + 5), "flops": n * m}
    if kind in ("sweep", "host"):
        return {"bytes": n * (2 * m + 6 * 5), "flops": 6 * n * m}
    if kind == "mapper":
        return {"bytes": n * (2 * m + 5 + m / 2), "flops": n * m}
    if kind == "unequal":
        mr = m + (case["above"] - case["below"]) / 2
        return {"bytes": n * ((m + mr) / 4 + 29), "flops": n * mr}
    out = 5 if kind == "submaze" else 4
    return {"bytes": n * (m / 2 + out), "flops": n * m}


# ---- the results, from their definitions -----------------------------------------

def _greedy(q, r, e, mr=None, t=None, y=None):
    """Obstacles of the paper's greedy, min(count, e + 1), for pairs q, r of
    shape (n, columns): the columns are walked one by one with the rows still
    free since each pair's last obstacle.  mr: reference lengths of their own
    (cells outside the read are then free where the lengths differ); t, y:
    the sub-maze decomposition."""
    n, m = q.shape
    cols = r.shape[1]
    pad = q.new_full((n, e), 255)
    wide = torch.cat([pad, q, q.new_full((n, cols - m + e), 255)], 1)
    free = torch.ones((n, 2 * e + 1), dtype=torch.bool, device=q.device)
    count = torch.zeros(n, dtype=torch.int64, device=q.device)
    part = torch.zeros_like(count)
    for j in range(cols):
        if t is not None and j % t == 0:
            count += part.clamp(max=y)
            part.zero_()
            free.fill_(True)
        base = wide[:, j:j + 2 * e + 1]
        ok = base == r[:, j:j + 1]
        if mr is not None:
            ok |= (base == 255) & (mr != m)[:, None]
        free &= ok
        dead = ~free.any(1)
        if mr is not None:
            dead &= j < mr
        if t is None:
            count += dead
        else:
            part += dead
        free |= dead[:, None]
    if t is not None:
        count += part.clamp(max=y)
    return count.clamp(max=e + 1)


def _distance(q, r, e):
    """min(edit distance, e + 1) by the banded table of the definition."""
    n, m = q.shape
    d = torch.arange(2 * e + 1, device=q.device)
    big = e + 1
    wide = torch.cat([r.new_full((n, e), 255), r, r.new_full((n, e), 255)], 1)
    row = (d - e).abs().clamp(max=big)
    row = torch.where(d >= e, row, big).expand(n, -1).clone()
    far = torch.full((n, 1), big, device=q.device)
    for i in range(1, m + 1):
        j = i + d - e
        miss = (wide[:, i - 1:i + 2 * e] != q[:, i - 1:i]).long()
        best = torch.minimum(row + miss, torch.cat([row[:, 1:], far], 1) + 1)
        best = torch.where(j == 0, i, best)
        best = torch.where((j < 0) | (j > m), 4 * big, best)
        row = torch.cummin(best - d, 1).values + d
        row = torch.where((j < 0) | (j > m), big, row).clamp(max=big)
    return row[:, e]


def _chunks(f, n, *sides):
    step = 1 << 19
    return torch.cat([f(*(x[a:a + step] for x in sides))
                      for a in range(0, n, step)])


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("batch", "sweep", "segments", "unequal", "submaze",
                    "distance", "mapper", "host"):
        return None
    g = _gen(seed)

    def both(obs, e):
        return (obs <= e).long(), obs

    if kind == "segments":
        out = []
        for n, m in ((case["n1"], case["m1"]), (case["n2"], case["m2"])):
            q, r = _fixed(g, n, m, _rates(g, n, 0.12), READ_MIX)
            e = _percent(m, case["percent"])
            out.append(both(_chunks(lambda a, b: _greedy(a, b, e), n,
                                    q.view(n, m), r.view(n, m)), e))
        return out
    n, m = case["n"], case["m"]
    e = case.get("e")
    if kind == "unequal":
        reads, refs, length, off = _windows(case, seed)
        top = m + case["above"]
        at = torch.arange(top, device="cuda")

        def windows(q, mr, o):
            idx = (o[:, None] + at).clamp(max=refs.numel() - 1)
            return _greedy(q, refs[idx], e, mr=mr)
        return both(_chunks(windows, n, reads.view(n, m), length, off), e)
    if kind == "batch":
        edits = torch.randint(0, 11, (n,), device="cuda", generator=g)
        q, r = _fixed(g, n, m, edits / 100 + 1e-6, EVEN_MIX)
    elif kind == "mapper":
        q, r = _fixed(g, n, m, _rates(g, n, 0.12), READ_MIX)
    else:
        q, r = _short(g, n, m)
    q, r = q.view(n, m), r.view(n, m)
    if kind in ("sweep", "host"):
        obs = [_chunks(lambda a, b: _greedy(a, b, k), n, q, r)
               for k in _sweep(m)]
        acc = [(o <= k).to(torch.uint8) for o, k in zip(obs, _sweep(m))]
        return torch.stack(acc), torch.stack(obs)
    if kind == "distance":
        return _chunks(lambda a, b: _distance(a, b, e), n, q, r)
    if kind == "submaze":
        obs = _chunks(lambda a, b: _greedy(a, b, e, t=case["t"], y=case["y"]),
                      n, q, r)
    else:
        obs = _chunks(lambda a, b: _greedy(a, b, e), n, q, r)
    acc, obs = both(obs, e)
    if kind == "mapper":
        return acc, obs, acc.sum()[None], None, None
    return acc, obs
