"""Host builds of the routes above 31 edits that do not depend on the bases:
a warp or a CTA per pair over all rows, and the index' way into them on
repeats and back, against the oracle."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_1910_09020_gb300 import synth

HERE = os.path.dirname(os.path.abspath(__file__))
EMU = os.path.join(HERE, "kernel_emu")
CSRC = os.path.join(os.path.dirname(HERE), "paper_1910_09020_gb300", "csrc")


@pytest.fixture(scope="module")
def emu():
    src = os.path.join(EMU, "emu_rows.cu")
    out = os.path.join(EMU, "_build", "libemu_rows.so")
    deps = [src] + [os.path.join(CSRC, f) for f in os.listdir(CSRC)
                    if f.endswith((".cuh", ".h"))]
    if (not os.path.exists(out)
            or any(os.path.getmtime(d) > os.path.getmtime(out)
                   for d in deps)):
        os.makedirs(os.path.dirname(out), exist_ok=True)
        nvcc = os.environ.get("NVCC", "nvcc")
        if not os.path.exists(nvcc) and os.path.exists(
                "/usr/local/cuda/bin/nvcc"):
            nvcc = "/usr/local/cuda/bin/nvcc"
        tmp = out + f".tmp{os.getpid()}"
        subprocess.check_call([nvcc, "-std=c++17", "-O2", "-gencode",
                               "arch=compute_103a,code=sm_103a", "-Xcompiler",
                               "-fPIC", "-shared", "-I", CSRC, src, "-o",
                               tmp])
        os.replace(tmp, out)
    lib = ctypes.CDLL(out)
    P, I = ctypes.c_void_p, ctypes.c_int
    lib.emu_rows.argtypes = [P, P, I, I, I]
    lib.emu_index_rows.argtypes = [P, P, I, I, I, I, P]
    lib.emu_column.argtypes = [P, P, I, I, I]
    lib.emu_rows_max_e.argtypes = [I]
    lib.emu_handed_over.argtypes = [P, P, I, I]
    lib.emu_first_pair.argtypes = [I, I, I]
    lib.emu_long_queued.argtypes = [I, I]
    return lib


def ptr(a):
    return ctypes.c_void_p(a.ctypes.data)


def packed(seq):
    return oracle.pack_reference(np.frombuffer(seq, np.uint8))


def noisy(rng, seq, rate):
    """seq with substitutions, insertions and deletions, of its length."""
    out = bytearray()
    for b in seq:
        u = rng.random()
        if u < rate / 3:
            out.append(b"ACGT"[rng.integers(4)])
        elif u < 2 * rate / 3:
            out += bytes([b, b"ACGT"[rng.integers(4)]])
        elif u >= rate:
            out.append(b)
    while len(out) < len(seq):
        out.append(b"ACGT"[rng.integers(4)])
    return bytes(out[:len(seq)])


def repeats(seed, m):
    """Pairs of repeats broken by errors on either side, and a repeat between
    random bases."""
    rng = np.random.default_rng(seed)
    units = [b"A", b"AC", bytes(b"ACGT"[i] for i in rng.integers(0, 4, 171))]
    out = []
    for unit in units:
        base = (unit * (m // len(unit) + 1))[:m]
        out.append((noisy(rng, base, 0.05), noisy(rng, base, 0.05)))
    q, _ = synth.pairs_fixed(seed, 0, 1, m, synth.rate_recipe(0.0))
    mixed = bytearray(q[0].tobytes())
    a = m // 3
    mixed[a:a + m // 4] = (b"AC" * m)[:m // 4]
    out.append((bytes(mixed), noisy(rng, bytes(mixed), 0.08)))
    return out


def plain(seed, m):
    out = []
    for k, rate in enumerate((0.002, 0.02, 0.2)):
        q, r = synth.pairs_fixed(seed + k, 0, 1, m, synth.rate_recipe(rate))
        out.append((q[0].tobytes(), r[0].tobytes()))
    out.append((out[0][0], out[0][0]))
    return out


@pytest.mark.parametrize("which", [0, 1, 2, 3])
def test_all_rows_match_oracle(emu, which):
    """Lengths around the words, the blocks of 1024 bases and the rings,
    thresholds from 0 to the largest of the rings."""
    top = emu.emu_rows_max_e(which)
    lengths = [1, 3, 4, 5, 31, 33, 100, 1023, 1024, 1025, 5000]
    if which == 0:
        lengths.append(9000)
    if which == 1:
        lengths.append(17000)
    for m in lengths:
        for k, (q, r) in enumerate(repeats(10 * m, m) + plain(20 * m, m)):
            if m > 1100 and k % 3:
                continue
            qw, rw = packed(q), packed(r)
            for E in sorted({0, 1, 40, m // 20, m // 3, top}):
                if E > top or (m > 1100 and E < 40):
                    continue
                want = oracle.filter_pair(q, r, E).obstacles
                got = emu.emu_rows(ptr(qw), ptr(rw), m, E, which)
                assert got == want, (which, m, E, k)


@pytest.mark.parametrize("ic,E", [(0, 817), (0, 1664), (1, 1665), (2, 6000)])
@pytest.mark.parametrize("calm", [1, 8])
def test_index_leaves_repeats_to_all_rows(emu, ic, E, calm):
    """The index route of a repeat goes over to all rows and, between random
    bases, comes back; the results are the oracle's."""
    m = {0: 6000, 1: 9000, 2: 14000}[ic]
    for k, (q, r) in enumerate(repeats(E, m) + plain(E, m)[2:3]):
        if ic == 2 and k in (0, 4):
            continue
        qw, rw = packed(q), packed(r)
        turns = ctypes.c_int()
        got = emu.emu_index_rows(ptr(qw), ptr(rw), m, E, ic, calm,
                                 ctypes.byref(turns))
        assert got == oracle.filter_pair(q, r, E).obstacles, (ic, E, k)
        if k in (0, 1, 3):
            assert turns.value > 0
        if k == 4 and got > 500:
            assert turns.value == 0


def test_index_thread_does_not_go_through_a_repeat(emu):
    """A column of a repeat is left to all rows (its thousands of starts are
    not gone through by one thread); one of random bases is not."""
    m, E = 4000, 1600
    for k, (q, r) in enumerate(repeats(5, m)[:2] + plain(6, m)[1:2]):
        qw, rw = packed(q), packed(r)
        many = [emu.emu_column(ptr(qw), ptr(rw), m, E, c)
                for c in range(1900, 2100)]
        assert (sum(many) > 100) if k < 2 else (sum(many) == 0)


def test_queue_takes_every_pair_above_511_edits(emu):
    """Also those above the index' thresholds, which would hold their batch's
    slot until the worker has left; and a worker's route for them."""
    for m in (600, 12000, 50000, 131072):
        for E in (31, 511, 512, 5920, 10016, 10017, 12000, 65000, 131071):
            e = min(E, m - 1)
            assert emu.emu_long_queued(m, E) == (e > 511), (m, E)
    for m, E in ((10100, 10017), (11000, 10999), (12000, 20000)):
        for q, r in repeats(m, m)[:1] + plain(m, m)[:2]:
            want = oracle.filter_pair(q, r, E).obstacles
            qw, rw = packed(q), packed(r)
            assert emu.emu_rows(ptr(qw), ptr(rw), m, E, 4) == want


def test_teams_hand_repeats_over_to_their_warp(emu):
    """A team's lane goes through a bounded number of survivors: a repeat is
    handed over within its first steps, a pair of random bases never is."""
    m, E = 6000, 800
    for k, (q, r) in enumerate(repeats(30, m)[:2] + plain(31, m)):
        qw, rw = packed(q), packed(r)
        at = emu.emu_handed_over(ptr(qw), ptr(rw), m, E)
        assert (0 < at < 200) if k < 2 else at == -1, (k, at)


@pytest.mark.parametrize("grid,sms", [(2128, 152), (1976, 152), (152, 152),
                                      (152 * 7, 76), (100, 152), (160, 152)])
def test_first_pairs_are_dealt_once(emu, grid, sms):
    """Each of the first pairs to one CTA, those of an SM's round spread over
    the launch."""
    got = [emu.emu_first_pair(b, grid, sms) for b in range(grid)]
    assert sorted(got) == list(range(grid))
    if grid >= 10 * sms:
        first = [b for b in range(grid) if got[b] < sms]
        assert max(sum(b // sms == k for b in first)
                   for k in range(grid // sms)) <= sms // 8


def test_worker_reads_sequences_by_ordinary_loads():
    """The serving worker outlives the kernels that write its pairs'
    sequences: its routes may not read them by the read-only path, which is
    defined only for memory that does not change while a kernel runs."""
    for name in ("ss_cws.cuh", "ss_cwx.cuh", "ss_server.cu"):
        with open(os.path.join(CSRC, name)) as f:
            code = "\n".join(line.split("//")[0] for line in f)
        assert "ldg(" not in code and ".nc" not in code, name
