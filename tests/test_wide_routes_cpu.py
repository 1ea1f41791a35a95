"""Host builds of the ring and index routes (thresholds above 31) against the
oracle, and the class table that chooses between them."""
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
    src = os.path.join(EMU, "emu_wide.cu")
    out = os.path.join(EMU, "_build", "libemu_wide.so")
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
    lib.emu_ring.argtypes = [P, P, I, I, I]
    lib.emu_index.argtypes = [P, P, I, I, I]
    lib.emu_wide_class.argtypes = [I, I, I]
    lib.emu_class_table.argtypes = [I, I]
    return lib


def ptr(a):
    return ctypes.c_void_p(a.ctypes.data)


def packed(seq):
    """Packed words of exactly the sequence's length, so that reading past
    them is noticed by address checkers."""
    return oracle.pack_reference(np.frombuffer(seq, np.uint8))


def some_pairs(seed, m):
    """Related and unrelated pairs, repeats of one and two bases (many rows
    alive at once), and a read against itself."""
    out = []
    for k, rate in enumerate((0.01, 0.08, 0.25)):
        q, r = synth.pairs_fixed(seed + k, 0, 1, m, synth.rate_recipe(rate))
        out.append((q[0].tobytes(), r[0].tobytes()))
    q, _ = synth.pairs_fixed(seed + 7, 0, 2, m, synth.rate_recipe(0.0))
    out.append((q[0].tobytes(), q[1].tobytes()))
    out.append((q[0].tobytes(), q[0].tobytes()))
    out.append((b"A" * m, (b"A" * (m // 2) + b"C" + b"A" * m)[:m]))
    out.append(((b"AC" * m)[:m], (b"AC" * (m // 3) + b"G" + b"CA" * m)[:m]))
    return out


@pytest.mark.parametrize("m", [1, 2, 3, 4, 5, 15, 16, 17, 31, 32, 33, 63, 64,
                               65, 96, 127, 160, 255, 256, 257, 448, 700])
def test_ring_route_matches_oracle(emu, m):
    """Lengths around the words, the last four columns and the ring's blocks
    (128 and 256 bases), small and clamped thresholds, every class."""
    for q, r in some_pairs(10 * m, m):
        qw, rw = packed(q), packed(r)
        for E in sorted({0, 1, 16, 31, 32, m // 10, m // 2, m + 3}):
            want = oracle.filter_pair(q, r, E).obstacles
            for rc in (0, 1, 2):
                if min(E, m - 1) <= emu.emu_class_table(4, rc):
                    got = emu.emu_ring(ptr(qw), ptr(rw), m, E, rc)
                    assert got == want, (m, E, rc, q, r)


@pytest.mark.parametrize("E", [32, 111, 112, 113, 303, 304, 305, 500, 815,
                               816])
def test_ring_route_at_class_bounds(emu, E):
    """Pairs of many ring blocks at thresholds up to the largest of each
    class (where the window, what is read past it and a block fill the
    ring)."""
    rc = sum(E > emu.emu_class_table(4, k) for k in (0, 1))
    for m in (1200, 6000):
        for q, r in some_pairs(E + m, m):
            qw, rw = packed(q), packed(r)
            want = oracle.filter_pair(q, r, E).obstacles
            assert emu.emu_ring(ptr(qw), ptr(rw), m, E, rc) == want, (E, m)


@pytest.mark.parametrize("ic", [0, 1, 2, 3])
def test_index_route_matches_oracle(emu, ic):
    """Every index shape, from thresholds far below to the largest its ring
    covers, lengths around the blocks (the small shape's ring of four
    blocks of 16 starts turns every 16 columns)."""
    top = 16 if ic == 3 else emu.emu_class_table(5, ic)
    block = (2048, 4096, 4096, 16)[ic]
    lengths = {1, 2, 5, 16, block - 1, block, block + 1, 3 * block + 7}
    if ic == 3:
        lengths |= {100, 700}
    if ic == 2:
        lengths = {1, 7, block - 1, block + 1}
    for m in sorted(lengths):
        for k, (q, r) in enumerate(some_pairs(100 * ic + m, m)):
            if m > 3000 and k not in (1, 3, 5):
                continue
            qw, rw = packed(q), packed(r)
            for E in sorted({0, 3, top // 7, top - 1, top}):
                if m > 3000 and E in (0, 3, top - 1):
                    continue
                want = oracle.filter_pair(q, r, E).obstacles
                got = emu.emu_index(ptr(qw), ptr(rw), m, E, ic)
                assert got == want, (ic, m, E, k)


def test_index_ring_past_its_blocks(emu):
    """A long pair whose window passes over every slot of the ring, at the
    largest threshold of the class."""
    m, E = 13000, 1664
    for q, r in some_pairs(900, m)[:4]:
        want = oracle.filter_pair(q, r, E).obstacles
        qw, rw = packed(q), packed(r)
        assert emu.emu_index(ptr(qw), ptr(rw), m, E, 0) == want


def test_class_table(emu):
    """Every (m, E') above 31 lands in a class whose bounds hold it."""
    T = emu.emu_class_table
    ring, index, cta, classes = (T(k, 0) for k in range(4))
    for m in (33, 100, 1024, 1025, 16384, 16385, 65537, 131072):
        for E in (16, 31, 32, 112, 113, 304, 305, 816, 817, 1664, 1665, 5920,
                  5921, 10016, 10017, 131071):
            for rmax in (15, 31):
                e = min(E, m - 1)
                c = emu.emu_wide_class(m, E, rmax)
                assert 0 <= c < classes
                if c < ring:
                    assert e <= rmax
                elif c < index:
                    assert rmax < e <= T(4, c - ring)
                elif c < cta:
                    assert T(4, 2) < e <= T(5, c - index)
                else:
                    assert e > 10016
    assert emu.emu_wide_class(131073, 32, 31) == -3
