"""The passes of 2^15 .. 2^20, joined in one launch or in a launch each, and those
of frames, at the edges of their ranges: the smallest batches, ragged batches
whose ring of workspace slots wraps, in place, buffers that are only 8-byte
aligned, repeated and overlapping-buffer calls, against the FP64 oracle."""
import numpy as np
import pytest

from paper_1505_08067_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(oracle, y, x_np, idx, direction, logn):
    ref = oracle.fft_select(x_np, idx, direction)
    assert np.max(oracle.rel_l2(y[torch.from_numpy(idx).cuda()].cpu().numpy(), ref)) <= 1e-6 * logn


# joined: the smallest batches that are, and larger ones; apart: one transform to
# the largest batches
@pytest.mark.parametrize("logn,batch", [(15, 391), (16, 193), (17, 97), (17, 131), (18, 49), (19, 25),
                                        (20, 12), (20, 13), (15, 1), (15, 3), (15, 64), (16, 7),
                                        (17, 1), (17, 75), (18, 1), (18, 47), (19, 1), (19, 3),
                                        (20, 1), (20, 11)])
@pytest.mark.parametrize("direction", [-1, 1])
def test_joined(gb, oracle, logn, batch, direction):
    joined = batch << logn >= 3 << 22
    n = 2 ** logn
    x_np = synth.uniform(700 + logn, batch, n)
    idx = np.unique([0, batch // 2, batch - 1])
    buf = torch.empty(batch * n + 1, dtype=torch.complex64, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    with gb.Plan(n, batch, direction) as p:
        d = p.describe()
        assert (d["joined"], d["apart"], p.launch_count) == ((1, 0, 1) if joined else (0, 1, 2))
        first = None
        for shift in (0, 1):  # 16-byte and 8-byte aligned input
            x = buf[shift:shift + batch * n].view(batch, n)
            x.copy_(torch.from_numpy(x_np))
            y = torch.empty(batch, n, dtype=torch.complex64, device="cuda")
            p.execute(x, y)
            first = y if first is None else first
            assert torch.equal(first, y)  # the counters are clean after each launch
        _check(oracle, first, x_np, idx, direction, logn)
        p.execute(x, x)
        gb.fft_plan_sync_status(p.handle, s)
        assert torch.equal(first, x)


@pytest.mark.parametrize("logn,batch", [(14, 1000), (21, 8)])
def test_not_joined(gb, logn, batch):
    with gb.Plan(2 ** logn, batch) as p:
        assert p.describe()["joined"] == 0 and p.describe()["apart"] == 0


@pytest.mark.parametrize("batch", [40, 193])
def test_partly_overlapping_buffers(gb, oracle, batch):
    """Output one transform after the input: the passes run apart, so that all
    of the input is read before any output is written."""
    logn = 16
    n = 2 ** logn
    x_np = synth.uniform(771, batch, n)
    buf = torch.empty((batch + 1) * n, dtype=torch.complex64, device="cuda")
    buf[:batch * n].copy_(torch.from_numpy(x_np).view(-1))
    with gb.Plan(n, batch) as p:
        assert p.describe()["joined"] == (1 if batch == 193 else 0)
        p.execute(buf[:batch * n], buf[n:])
        torch.cuda.synchronize()
    _check(oracle, buf[n:].view(batch, n), x_np, np.array([0, 1, batch - 1]), -1, logn)


def test_two_plans_on_two_streams(gb, oracle):
    logn, batch = 17, 100
    n = 2 ** logn
    xs = [torch.from_numpy(synth.uniform(780 + i, batch, n)).cuda() for i in range(2)]
    streams = [torch.cuda.Stream() for _ in xs]
    torch.cuda.synchronize()
    with gb.Plan(n, batch) as p, gb.Plan(n, batch) as q:
        want = [p.execute(x) for x in xs]
        torch.cuda.synchronize()
        got = [torch.empty_like(x) for x in xs]
        for _ in range(8):
            for plan, x, y, s in zip((p, q), xs, got, streams):
                plan.execute(x, y, stream=s)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(want, got))


def test_one_frame_plan_on_two_streams(gb):
    """Frame plans have no workspace: executions on several streams may overlap."""
    shape, batch = (512, 256), 100
    xs = [torch.from_numpy(synth.uniform(790 + i, batch, shape[0] * shape[1])).cuda()
          .view((batch,) + shape) for i in range(2)]
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    with gb.Plan(shape, batch) as p:
        assert p.describe()["joined"] == 1
        want = [p.execute(x, stream=streams[0]) for x in xs]
        torch.cuda.synchronize()
        got = [torch.empty_like(x) for x in xs]
        for _ in range(8):
            for x, y, s in zip(xs, got, streams):
                p.execute(x, y, stream=s)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(want, got))
        gb.fft_plan_sync_status(p.handle, streams[0].cuda_stream)
        # a graph of one execution beside the other on a stream
        got = [torch.empty_like(x) for x in xs]
        for _ in range(4):
            p.execute_graph(xs[1], got[1], stream=streams[1])
            p.execute(xs[0], got[0], stream=streams[0])
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(want, got))
        gb.fft_plan_sync_status(p.handle, streams[0].cuda_stream)


# joined frames, then frames whose passes are launches of the short-line kernels
@pytest.mark.parametrize("shape,batch", [((16, 16), 49153), ((32, 64), 6145), ((64, 128), 1537),
                                         ((512, 16), 1537), ((128, 32), 3073), ((1024, 512), 25),
                                         ((2048, 16), 385), ((256, 256), 193), ((512, 1024), 24),
                                         ((8, 4), 3), ((16, 16), 1), ((16, 16), 8193), ((64, 64), 3),
                                         ((32, 64), 1031), ((64, 128), 257), ((1024, 16), 1),
                                         ((512, 16), 257), ((256, 8192), 1), ((16, 4096), 33),
                                         ((1024, 512), 5), ((2048, 16), 65), ((2048, 2048), 1)])
@pytest.mark.parametrize("direction", [-1, 1])
def test_joined_frames(gb, oracle, shape, batch, direction):
    """Frames smaller than a tile with a ragged last one, frames of one tile and
    of many, both tile sizes, both ends of the length ranges."""
    n = shape[0] * shape[1]
    x_np = synth.uniform(800 + shape[0], batch, n).reshape((batch,) + shape)
    idx = np.unique([0, batch // 2, batch - 1])
    buf = torch.empty(batch * n + 1, dtype=torch.complex64, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    with gb.Plan(shape, batch, direction) as p:
        d = p.describe()
        assert d["joined"] == (1 if batch * n >= 3 << 22 else 0) and d["kernels"][1]["lines"] == 1
        first = None
        for shift in (0, 1):
            x = buf[shift:shift + batch * n].view((batch,) + shape)
            x.copy_(torch.from_numpy(x_np))
            y = torch.full_like(x, float("nan"))
            p.execute(x, y)
            first = y if first is None else first
            assert torch.equal(first, y)
        p.execute(x, x)
        gb.fft_plan_sync_status(p.handle, s)
        assert torch.equal(first, x)
    ref = oracle.fft2d(x_np[idx], direction).reshape(len(idx), n)
    got = first[torch.from_numpy(idx).cuda()].cpu().numpy().reshape(len(idx), n)
    assert np.max(oracle.rel_l2(got, ref)) <= 1e-6 * np.log2(n)


@pytest.mark.parametrize("shape,batch", [((512, 16), 1535), ((8, 4096), 800), ((4096, 512), 10),
                                         ((64, 2048), 100), ((64, 16384), 30)])
def test_frames_not_joined(gb, shape, batch):
    with gb.Plan(shape, batch) as p:
        assert p.describe()["joined"] == 0 and p.launch_count == 2


@pytest.mark.parametrize("logn", [15, 18, 20])
def test_joined_sub_batches(gb, oracle, logn):
    """A batch above 2^28 elements: the last sub-batch is a few transforms through
    the ring and the counters that the whole one before left, and the same from a graph."""
    n, chunk = 2 ** logn, 2 ** (28 - logn)
    batch = chunk + 3
    g = torch.Generator(device="cuda")
    g.manual_seed(logn)
    x = torch.view_as_complex(torch.rand((batch, n, 2), generator=g, device="cuda").mul_(2).sub_(1))
    s = torch.cuda.current_stream().cuda_stream
    idx = np.array([0, chunk - 1, chunk, batch - 1])
    with gb.Plan(n, batch) as p:
        d = p.describe()
        assert (d["joined"], d["chunk_batch"]) == (1, chunk)
        y = p.execute(x)
        gb.fft_plan_sync_status(p.handle, s)
        rows = x[torch.from_numpy(idx).cuda()]
        _check(oracle, y, np.broadcast_to(rows[0].cpu().numpy(), (1, n)), np.array([0]), -1, logn)
        with gb.Plan(n, len(idx)) as q:  # apart
            assert torch.equal(q.execute(rows), y[torch.from_numpy(idx).cuda()])
        z = torch.empty_like(x)
        p.execute_graph(x, z)
        p.execute(x, x)
        gb.fft_plan_sync_status(p.handle, s)
        assert torch.equal(z, y) and torch.equal(x, y)
