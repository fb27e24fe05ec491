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
    f = ctypes.CDLL(lib)
    f.join_run.restype = f.join_run_frames.restype = ctypes.c_int64
    f.join_run.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int64, ctypes.c_int, ctypes.c_int64,
                           ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_char_p, ctypes.c_size_t]
    f.join_run_frames.argtypes = [ctypes.c_int64, ctypes.c_int, ctypes.c_int, ctypes.c_int,
                                  ctypes.c_void_p, ctypes.c_void_p, ctypes.c_char_p, ctypes.c_size_t]
    return f


# every transform length in every tile it runs in; one transform, a ring that is
# reused, a lag of several transforms, no reuse (lag in tiles: 8 to 128 a transform)
@pytest.mark.parametrize("logn,tile,batch,lag,ring",
                         [(15, 12, 7, 19, 4), (15, 12, 1, 40, 1), (16, 12, 3, 16, 2),
                          (17, 12, 1, 32, 1), (17, 13, 3, 33, 4), (18, 12, 1, 64, 1),
                          (18, 13, 3, 32, 2), (19, 13, 2, 64, 2), (20, 13, 1, 128, 1),
                          (20, 14, 1, 64, 1)])
@pytest.mark.parametrize("direction", [-1, 1])
def test_joined(oracle, joined, logn, tile, batch, lag, ring, direction):
    x = synth.uniform(60 + logn, batch, 2 ** logn)
    y = np.zeros_like(x)
    msg = ctypes.create_string_buffer(256)
    n = joined.join_run(logn, tile, batch, int(direction > 0), lag, ring, x.ctypes.data, y.ctypes.data, msg, 256)
    assert n == 0, msg.value.decode()
    assert np.max(oracle.rel_l2(y, oracle.fft(x, direction))) <= 1e-6 * logn


# every column length and row length, frames smaller than a tile with a ragged
# last one, both tile sizes
@pytest.mark.parametrize("lr,lc,batch", [(4, 4, 37), (5, 6, 7), (6, 5, 3), (7, 7, 2), (8, 8, 2),
                                         (9, 4, 3), (10, 5, 2), (11, 6, 1), (8, 9, 1), (5, 10, 2),
                                         (9, 9, 1), (10, 4, 5)])
@pytest.mark.parametrize("direction", [-1, 1])
def test_joined_frames(oracle, joined, lr, lc, batch, direction):
    x = synth.uniform(80 + lr, batch, 2 ** (lr + lc)).reshape(batch, 2 ** lr, 2 ** lc)
    y = np.zeros_like(x)
    msg = ctypes.create_string_buffer(256)
    n = joined.join_run_frames(batch, lr, lc, int(direction > 0), x.ctypes.data, y.ctypes.data, msg, 256)
    assert n == 0, msg.value.decode()
    ref = oracle.fft2d(x, direction).reshape(batch, -1)
    assert np.max(oracle.rel_l2(y.reshape(batch, -1), ref)) <= 1e-6 * (lr + lc)


@pytest.mark.parametrize("logl,cols,batch", [(3, 0, 600), (4, 0, 257), (5, 0, 3), (6, 0, 65), (7, 0, 33),
                                             (8, 0, 17), (9, 0, 9), (10, 0, 5), (11, 0, 3), (3, 64, 9), (5, 16, 9), (6, 128, 1), (7, 4, 9),
                                             (8, 32, 1), (9, 8, 3), (10, 16, 1), (11, 8, 1)])
@pytest.mark.parametrize("per_line", [False, True])
def test_conv_tiles(oracle, joined, logl, cols, batch, per_line):
    """Fast convolution of lines (cols = 0) and of frame columns, a ragged last tile."""
    n = 2 ** logl
    f = joined.conv_run
    f.restype = ctypes.c_int64
    f.argtypes = [ctypes.c_int64, ctypes.c_int, ctypes.c_int, ctypes.c_int64, ctypes.c_float] + \
        [ctypes.c_void_p] * 3 + [ctypes.c_char_p, ctypes.c_size_t]
    lines = (cols or batch) if per_line else 1
    x = synth.uniform(90 + logl, batch, n * max(1, cols)).reshape(batch, n, max(1, cols))
    h = synth.uniform(190 + logl, lines, n)  # a filter per line
    hl = np.ascontiguousarray(h.T) if cols else h  # columns: laid out like a frame
    y = np.zeros_like(x)
    msg = ctypes.create_string_buffer(256)
    e = f(batch, logl, cols, lines, 1.0 / n, hl.ctypes.data, x.ctypes.data, y.ctypes.data, msg, 256)
    assert e == 0, msg.value.decode()
    H = (h.T[None] if cols else h[:, :, None]).astype(np.complex128)
    ref = np.fft.ifft(np.fft.fft(x.astype(np.complex128), axis=1) * H, axis=1)
    assert np.linalg.norm(y - ref) <= 2e-6 * logl * np.linalg.norm(ref)
