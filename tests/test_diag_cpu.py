"""Host build of the distance kernel by diagonals, its loop and its arrays as
on the GPU, against the oracle."""
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
    src = os.path.join(EMU, "emu_diag.cu")
    out = os.path.join(EMU, "_build", "libemu_diag.so")
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
    lib.emu_diag.argtypes = [P, P, I, I, I, I]
    return lib


@pytest.mark.parametrize("m", [1, 2, 15, 16, 17, 40, 100, 333, 700])
def test_diagonals_match_oracle(emu, m):
    """Both teams of the launches (8 lanes up to 63 edits, 32 up to 511), at
    thresholds either side of the switch, of the distance and of the length."""
    for k, rate in enumerate((0.0, 0.02, 0.1, 0.4)):
        q, r = synth.pairs_fixed(900 + m + k, 0, 1, m, synth.rate_recipe(rate))
        a, b = q[0].tobytes(), r[0].tobytes()
        ed = oracle.edit_distance(a, b)
        qw, rw = (oracle.pack_reference(np.frombuffer(x, np.uint8))
                  for x in (a, b))
        for E in sorted({0, 1, 2, 3, 8, 62, 63, 64, 65, 510, 511, m,
                         max(ed - 1, 0), ed, ed + 1}):
            if E > 511:
                continue
            for nt, top in ((8, 63), (32, 511)):
                if E <= top:
                    got = emu.emu_diag(ctypes.c_void_p(qw.ctypes.data),
                                       ctypes.c_void_p(rw.ctypes.data), m, E,
                                       nt, top)
                    assert got == min(ed, E + 1), (m, E, nt, ed)
