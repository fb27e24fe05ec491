"""CPU replay of the joined two-pass kernel (tests/emu/join_harness.cpp): every
access checked, every wait for earlier tickets only, and the transform within
the FP32 tolerance of the FP64 oracle, against which the two-launch form of the
same plans is replayed in test_emulated_addressing.py."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1505_08067_gb300 import synth

HERE = os.path.join(os.path.dirname(os.path.abspath(__file__)), "emu")
CSRC = os.path.join(os.path.dirname(os.path.dirname(HERE)), "paper_1505_08067_gb300", "csrc")


@pytest.fixture(scope="session")
def joined():
    lib, src = os.path.join(HERE, "_join.so"), os.path.join(HERE, "join_harness.cpp")
    deps = [src] + [os.path.join(CSRC, f) for f in ("fft_join.h", "fft_stage.h", "fft_core.h")]
    if not os.path.exists(lib) or os.path.getmtime(lib) < max(map(os.path.getmtime, deps)):
        tmp = lib + f".tmp{os.getpid()}"
        subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC",
                        "-Wno-unknown-pragmas", "-I" + CSRC, "-o", tmp, src], check=True)
        os.replace(tmp, lib)
    f = ctypes.CDLL(lib).join_run
    f.restype = ctypes.c_int64
    f.argtypes = [ctypes.c_int, ctypes.c_int64, ctypes.c_int, ctypes.c_int, ctypes.c_int,
                  ctypes.c_void_p, ctypes.c_void_p, ctypes.c_char_p, ctypes.c_size_t]
    return f


# one transform, a ring that is reused, a lag of several transforms, no reuse
@pytest.mark.parametrize("logn,batch,lag,ring", [(15, 7, 2, 3), (15, 1, 4, 1), (16, 3, 1, 2),
                                                 (17, 3, 2, 3), (18, 3, 1, 2), (19, 2, 1, 2),
                                                 (20, 1, 1, 1)])
@pytest.mark.parametrize("direction", [-1, 1])
def test_joined(oracle, joined, logn, batch, lag, ring, direction):
    x = synth.uniform(60 + logn, batch, 2 ** logn)
    y = np.zeros_like(x)
    msg = ctypes.create_string_buffer(256)
    n = joined(logn, batch, int(direction > 0), lag, ring, x.ctypes.data, y.ctypes.data, msg, 256)
    assert n == 0, msg.value.decode()
    assert np.max(oracle.rel_l2(y, oracle.fft(x, direction))) <= 1e-6 * logn
