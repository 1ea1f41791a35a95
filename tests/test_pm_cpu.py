"""Host builds of the pair-major batches' bit-sliced walks (sub-maze mode,
capped distance) against the oracle."""
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
    src = os.path.join(EMU, "emu_pm.cu")
    out = os.path.join(EMU, "_build", "libemu_pm.so")
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
        subprocess.check_call([nvcc, "-std=c++17", "-O1", "-Xcicc", "-O0",
                               "-Xptxas", "-O0", "-gencode",
                               "arch=compute_103a,code=sm_103a", "-Xcompiler",
                               "-fPIC", "-shared", "-I", CSRC, src, "-o",
                               tmp])
        os.replace(tmp, out)
    lib = ctypes.CDLL(out)
    P, I = ctypes.c_void_p, ctypes.c_int
    lib.emu_pm.argtypes = [P, P, ctypes.c_int64, I, I, I, I, I, P]
    lib.emu_transpose.argtypes = [P]
    return lib


def ptr(a):
    return ctypes.c_void_p(a.ctypes.data)


def batch(seed, n, m):
    """n pairs, a third each related closely, loosely and not at all."""
    parts = [synth.pairs_fixed(seed + k, 0, n, m, synth.rate_recipe(rate))
             for k, rate in enumerate((0.04, 0.2))]
    q, r = parts[0][0].copy(), parts[0][1].copy()
    q[1::3], r[1::3] = parts[1][0][1::3], parts[1][1][1::3]
    r[2::3] = parts[1][1][:len(r[2::3])]
    pack = lambda x: np.concatenate(  # noqa: E731
        [oracle.pack_reference(row) for row in x])
    return q, r, pack(q), pack(r)


def run(emu, qw, rw, n, m, E, what, t=0, y=0):
    out = np.full(n, -7, np.int32)
    emu.emu_pm(ptr(qw), ptr(rw), n, m, E, what, t, y, ptr(out))
    return out


def test_transpose(emu):
    a = np.random.default_rng(3).integers(0, 1 << 32, 32, dtype=np.uint32)
    b = a.copy()
    emu.emu_transpose(ptr(b))
    bits = (a[:, None] >> np.arange(32, dtype=np.uint32)) & 1
    want = (bits.T.astype(np.uint64) << np.arange(32, dtype=np.uint64)).sum(1)
    assert (b == want).all()


@pytest.mark.parametrize("m", [1, 3, 4, 5, 15, 16, 17, 31, 33, 64, 100])
def test_walks_match_oracle(emu, m):
    """Every threshold it takes, lengths around a block, a word and below E, a group
    that is not full."""
    n = 41
    q, r, qw, rw = batch(m, n, m)
    eds = np.array([oracle.edit_distance(q[i].tobytes(), r[i].tobytes())
                    for i in range(n)])
    for E in range(32):
        # one sub-maze over the whole pair is the exact filter
        want = oracle.filter_batch(q, r, m, E)[1]
        got = run(emu, qw, rw, n, m, E, 0, m, E + 1)
        assert (got == want).all(), (m, E)
        got = run(emu, qw, rw, n, m, E, 1)
        assert (got == np.minimum(eds, E + 1)).all(), (m, E)


@pytest.mark.parametrize("t,y", [(1, 1), (8, 3), (31, 2), (200, 40)])
def test_submaze_matches_oracle(emu, t, y):
    n, m = 33, 90
    q, r, qw, rw = batch(7, n, m)
    for E in (0, 1, 5, 12, 31):
        want = [oracle.filter_submaze(q[i].tobytes(), r[i].tobytes(), E, t,
                                      y).obstacles for i in range(n)]
        assert (run(emu, qw, rw, n, m, E, 0, t, y) == want).all(), E
