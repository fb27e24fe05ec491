"""Device-side failure detection without a fault: the kernels' bounded
mbarrier wait, run on a barrier that nothing completes (fft_wait_selftest),
gives up after its poll limit, reports it through a status word the host
reads, and leaves the device usable: a plan executed afterwards still matches
the FP64 oracle."""
import time

import numpy as np
import pytest

from paper_1505_08067_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_wait_gives_up_and_device_stays_usable(gb, oracle):
    for polls in (1, 64, 4096, 1 << 16):
        t0 = time.perf_counter()
        assert gb.fft_wait_selftest(polls) == 1
        assert time.perf_counter() - t0 < 5.0
    for polls in (0, 2 ** 22 + 1):
        with pytest.raises(gb.GbfftError):
            gb.fft_wait_selftest(polls)
    # staged kernels (2^13) and a two-pass plan run normally afterwards
    for n, batch in ((8192, 33), (2 ** 20, 2)):
        x_np = synth.uniform(7100 + batch, batch, n)
        x = torch.from_numpy(x_np).cuda()
        with gb.Plan(n, batch) as p:
            y = p.execute(x)
            gb.fft_plan_sync_status(p.handle, torch.cuda.current_stream().cuda_stream)
        err = oracle.rel_l2(y.cpu().numpy(), oracle.fft(x_np))
        assert np.max(err) <= 1e-6 * np.log2(n), float(np.max(err))


JOINED = [((2 ** 15,), 391), ((2 ** 17,), 131), ((2 ** 20,), 13), ((16, 16), 49153), ((1024, 512), 25)]


def _joined(gb, shape, batch):
    torch.manual_seed(batch)
    x = torch.randn((batch,) + shape, dtype=torch.complex64, device="cuda")
    p = gb.Plan(shape if len(shape) > 1 else shape[0], batch)
    assert p.describe()["joined"] == 1
    return p, x, p.execute(x)


@pytest.mark.parametrize("shape,batch", JOINED)
@pytest.mark.parametrize("lost", [1, 7])
def test_joined_wait_gives_up(gb, shape, batch, lost):
    """The first `lost` tiles are never computed: what depends on them gives up, in
    whichever block it falls to, the launch ends, the host reads it from the
    status word, and the next execution starts from clean counters."""
    s = torch.cuda.current_stream().cuda_stream
    p, x, want = _joined(gb, shape, batch)
    with p:
        y = torch.empty_like(x)
        for polls in (1, 64, 4096):
            t0 = time.perf_counter()
            gb.fft_join_selftest(p.handle, x.data_ptr(), y.data_ptr(), lost, polls, s)
            with pytest.raises(gb.GbfftError) as e:
                gb.fft_plan_sync_status(p.handle, s)
            assert e.value.status == gb.FFT_ERR_TIMEOUT and time.perf_counter() - t0 < 5.0
            y.fill_(float("nan"))
            p.execute(x, y)
            gb.fft_plan_sync_status(p.handle, s)
            assert torch.equal(y, want)
        for polls in (0, 2 ** 21 + 1):
            with pytest.raises(gb.GbfftError):
                gb.fft_join_selftest(p.handle, x.data_ptr(), y.data_ptr(), lost, polls, s)
    with gb.Plan(1024, 4) as q, pytest.raises(gb.GbfftError):
        gb.fft_join_selftest(q.handle, x.data_ptr(), y.data_ptr(), lost, 64, s)


@pytest.mark.parametrize("shape,batch", JOINED)
def test_joined_counters_not_its_own(gb, shape, batch):
    """A launch that finds every tile handed out computes nothing and waits for
    nothing: it is reported, once, and the plan is as new."""
    s = torch.cuda.current_stream().cuda_stream
    p, x, want = _joined(gb, shape, batch)
    with p:
        y = torch.empty_like(x)
        for handed_out in (2 * x.numel(), 2 ** 31):
            gb.fft_join_selftest(p.handle, x.data_ptr(), y.data_ptr(), handed_out, 64, s)
            with pytest.raises(gb.GbfftError) as e:
                gb.fft_plan_sync_status(p.handle, s)
            assert e.value.status == gb.FFT_ERR_CUDA
            y.fill_(float("nan"))
            p.execute(x, y)
            gb.fft_plan_sync_status(p.handle, s)
            assert torch.equal(y, want)


@pytest.mark.parametrize("shape,batch", [((2 ** 15,), 391), ((2 ** 18,), 49)])
def test_cleared_counters_before_the_next_execution(gb, shape, batch):
    """fft_plan_sync_status returns with the counters cleared: an execution that follows
    at once, on a stream that waits for no other, finds them so."""
    p, x, want = _joined(gb, shape, batch)
    outs = [torch.full_like(x, float("nan")) for _ in range(8)]
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with p:
        for i in range(40):
            y = outs[i % 8]
            gb.fft_join_selftest(p.handle, x.data_ptr(), y.data_ptr(), 2 ** 31, 64, a.cuda_stream)
            with pytest.raises(gb.GbfftError):
                gb.fft_plan_sync_status(p.handle, a.cuda_stream)
            gb.fft_execute(p.handle, x.data_ptr(), y.data_ptr(), b.cuda_stream)
            gb.fft_plan_sync_status(p.handle, b.cuda_stream)
        assert all(torch.equal(y, want) for y in outs)


def test_joined_selftest_is_not_captured(gb):
    """Refused in a capture, which stays valid."""
    p, x, want = _joined(gb, (2 ** 15,), 391)
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    with p:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            s = torch.cuda.current_stream().cuda_stream
            with pytest.raises(gb.GbfftError) as e:
                gb.fft_join_selftest(p.handle, x.data_ptr(), y.data_ptr(), 1, 64, s)
            gb.fft_execute(p.handle, x.data_ptr(), y.data_ptr(), s)
        assert e.value.status == gb.FFT_ERR_INVALID_ARG
        g.replay()
        gb.fft_plan_sync_status(p.handle, torch.cuda.current_stream().cuda_stream)
        assert torch.equal(y, want)
