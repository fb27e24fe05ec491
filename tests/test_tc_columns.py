"""Tensor-core plans of 2^15 .. 2^20 points execute their row passes on column
tiles (the tcgen05 kernel's modes 1 to 3) instead of the six steps, without the
transposes (BF16x3, complex32) or without the first and the last: the CPU replay
with every access checked, and the GPU against the FP64 oracle, within the class
tolerances of the six-step form."""
import ctypes

import numpy as np
import pytest

from emu import emu
from paper_1505_08067_gb300 import synth

# relative L2 of the class above 2^14 (see test_tc_gpu.py)
TOL = {1: lambda n: 2e-3, 2: lambda n: 7e-3, 3: lambda n: 5e-6 * np.log2(n), 4: lambda n: 2e-3}


@pytest.mark.parametrize("logn,precision,direction", [(15, 1, -1), (15, 3, 1), (16, 2, 1), (17, 3, -1),
                                                      (18, 1, 1), (20, 1, -1)])
def test_replay(oracle, logn, precision, direction):
    n, batch = 2 ** logn, 2 if logn < 18 else 1
    lib = emu.load()
    lib.emu_tc_cols_run.restype = ctypes.c_int64
    lib.emu_tc_cols_run.argtypes = [ctypes.c_int64, ctypes.c_int64, ctypes.c_int, ctypes.c_int,
                                    ctypes.c_void_p, ctypes.c_void_p, ctypes.c_char_p, ctypes.c_size_t]
    x = synth.uniform(300 + logn, batch, n)
    y = np.zeros_like(x)
    msg = ctypes.create_string_buffer(256)
    e = lib.emu_tc_cols_run(n, batch, direction, precision, x.ctypes.data, y.ctypes.data, msg, 256)
    assert e == 0, msg.value.decode()
    assert np.max(oracle.rel_l2(y, oracle.fft(x, direction))) <= TOL[precision](n)


@pytest.mark.gpu
@pytest.mark.parametrize("logn,batch", [(15, 1), (15, 83), (16, 41), (17, 3), (18, 11), (19, 1), (20, 5)])
@pytest.mark.parametrize("precision", [1, 2, 3, 4])
def test_columns(gb, oracle, logn, batch, precision):
    """One transform, and more tiles than the persistent grid; out of place, in
    place, and from an input that no tensor map can describe."""
    torch = pytest.importorskip("torch")
    n, direction = 2 ** logn, -1 if batch % 2 else 1
    x_np = synth.uniform(320 + logn, batch, n)
    if precision == 4:
        h = np.ascontiguousarray(np.stack([x_np.real, x_np.imag], -1).astype(np.float16))
        x_np = h[..., 0].astype(np.float32) + 1j * h[..., 1].astype(np.float32)
        data, dtype, bits = torch.from_numpy(h).cuda().view(-1), torch.complex32, torch.int32
    else:
        data, dtype, bits = torch.view_as_real(torch.from_numpy(x_np).cuda()).reshape(-1), torch.complex64, torch.int64
    buf = torch.empty(2 * (batch * n + 1), dtype=data.dtype, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    idx = np.unique([0, batch // 2, batch - 1])
    ref = oracle.fft_select(x_np.astype(np.complex64), idx, direction)

    def error(y):
        v = torch.view_as_real(y.view(batch, n)[torch.from_numpy(idx).cuda()]) if precision != 4 else \
            y.view(torch.float16).view(batch, n, 2)[torch.from_numpy(idx).cuda()]
        v = v.float().cpu().numpy()
        return np.max(oracle.rel_l2(v[..., 0] + 1j * v[..., 1], ref))

    with gb.Plan(n, batch, direction, precision) as p:
        assert p.describe()["tc_columns"] == 1 and p.launch_count == (2 if precision > 2 else 3)
        for shift in (0, 1):
            flat = buf[2 * shift:2 * (shift + batch * n)]
            flat.copy_(data)
            x = flat.view(dtype)
            y = torch.empty(batch * n, dtype=dtype, device="cuda")
            gb.fft_execute(p.handle, x.data_ptr(), y.data_ptr(), s)
            gb.fft_plan_sync_status(p.handle, s)
            assert error(y) <= TOL[precision](n), shift
        gb.fft_execute(p.handle, x.data_ptr(), x.data_ptr(), s)
        gb.fft_plan_sync_status(p.handle, s)
        assert torch.equal(x.view(bits), y.view(bits))


@pytest.mark.gpu
@pytest.mark.parametrize("logn,batch", [(15, 83), (16, 5), (17, 3), (18, 11), (19, 1), (20, 5)])
@pytest.mark.parametrize("precision", [1, 2, 3, 4])
def test_six_steps(gb, oracle, logn, batch, precision):
    """The six-step form of the same lengths (the generic option) against the oracle;
    FP16 and BF16 with complex64 data keep its bits on column tiles."""
    torch = pytest.importorskip("torch")
    n, direction = 2 ** logn, 1 if batch % 2 else -1
    x_np = synth.uniform(340 + logn, batch, n)
    x = torch.from_numpy(x_np).cuda()
    if precision == 4:
        h = torch.view_as_real(x).half().contiguous()
        x, x_np = torch.view_as_complex(h), torch.view_as_complex(h.float()).cpu().numpy()
    with gb.Plan(n, batch, direction, precision, generic=1) as p, gb.Plan(n, batch, direction, precision) as q:
        assert p.describe()["tc_columns"] == 0 and q.describe()["tc_columns"] == 1
        y, z = p.execute(x), q.execute(x)
        torch.cuda.synchronize()
    if precision <= 2:
        assert torch.equal(y.view(torch.int64), z.view(torch.int64))
    ref = oracle.fft_select(x_np, np.array([0, batch - 1]), direction)
    v = torch.view_as_real(y).float().cpu().numpy()[[0, batch - 1]]
    assert np.max(oracle.rel_l2(v[..., 0] + 1j * v[..., 1], ref)) <= TOL[precision](n)
