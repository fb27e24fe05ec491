"""Which streams a joined frame plan has tile counters for: csrc/join_owner.h under
threads on the CPU, and the streams of a real plan."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1505_08067_gb300", "csrc")


@pytest.mark.parametrize("threads,ids", [(1, 1), (1, 9), (4, 3), (8, 4), (8, 7)])
def test_owners(tmp_path, threads, ids):
    lib = str(tmp_path / "owners.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-pthread", "-I" + CSRC, "-o", lib,
                    os.path.join(HERE, "emu", "owner_harness.cpp")], check=True)
    assert ctypes.CDLL(lib).owners_run(threads, ids, 200) == 0


@pytest.mark.gpu
def test_frame_plan_streams(gb):
    """A host execution and a warm-up on a side stream leave sets for two more
    streams, which join; the fifth runs a launch per pass; all at once, in any
    order, with one result."""
    torch = pytest.importorskip("torch")
    shape, batch = (512, 256), 100
    torch.manual_seed(3)
    x = torch.randn((batch,) + shape, dtype=torch.complex64, device="cuda")
    streams = [torch.cuda.Stream() for _ in range(4)]
    host = x.cpu().pin_memory()
    back = torch.empty_like(host).pin_memory()
    tmp = torch.empty_like(x)
    with gb.Plan(shape, batch) as p:
        p.execute_host(host, back, tmp, tmp)
        torch.cuda.synchronize()
        want = p.execute(x, stream=streams[0])
        torch.cuda.synchronize()
        assert torch.equal(back, want.cpu())
        outs = [torch.empty_like(x) for _ in streams]
        for k, (s, y) in enumerate(zip(streams, outs)):  # nothing handed out: an execution
            run = lambda: gb.fft_join_selftest(p.handle, x.data_ptr(), y.data_ptr(), 0, 2 ** 21, s.cuda_stream)
            if k < 3:
                run()
                torch.cuda.synchronize()
                assert torch.equal(y, want)
            else:
                with pytest.raises(gb.GbfftError):
                    run()
        for y in outs:
            y.zero_()
        torch.cuda.synchronize()
        for _ in range(8):
            for s, y in zip(streams, outs):
                p.execute(x, y, stream=s)
        p.execute_host(host, back, tmp, tmp)
        torch.cuda.synchronize()
        assert all(torch.equal(y, want) for y in outs) and torch.equal(back, want.cpu())
        gb.fft_plan_sync_status(p.handle, streams[0].cuda_stream)
