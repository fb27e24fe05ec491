"""One transform, one result: every entry point runs an FP32 shape with the same
arithmetic, so a job's output has the bits of fft_execute with default options,
whatever else is waiting."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _bits(t):
    return t.view(torch.int64)


def _case(gb, logn, batches, direction):
    """Inputs, what fft_execute gives for them, and outputs inside guard elements."""
    n = 2 ** logn
    torch.manual_seed(logn)
    xs = [torch.randn(b * n, dtype=torch.complex64, device="cuda") for b in batches]
    want = []
    for x, b in zip(xs, batches):
        with gb.Plan(n, b, direction) as p:
            want.append(p.execute(x))
    outs = [torch.full((b * n + 1,), 7.0 + 7.0j, dtype=torch.complex64, device="cuda") for b in batches]
    torch.cuda.synchronize()
    return n, xs, want, outs


def _check(xs, want, outs):
    torch.cuda.synchronize()
    for x, w, y in zip(xs, want, outs):
        assert torch.equal(_bits(y[:-1]), _bits(w)) and y[-1].item() == 7.0 + 7.0j


@pytest.mark.parametrize("logn", list(range(1, 21)) + [21])
@pytest.mark.parametrize("direction", [-1, 1])
def test_server(gb, logn, direction):
    """A job alone, and jobs of several sizes in one held burst (lengths up to 2^14:
    one coalesced launch, here in more than one table of jobs), with ragged tiles."""
    t = max(1, 4096 >> logn)
    batches = [1, t, t + 1, 3 * t - 1 or 1, 2] * (14 if logn <= 14 else 1)
    n, xs, want, outs = _case(gb, logn, batches, direction)
    srv = gb.fft_server_create(memory_budget_bytes=4 << 30)
    try:
        submit = lambda x, y, b: gb.fft_server_submit(srv, n, b, direction, 0, x.data_ptr(), y.data_ptr())
        for x, y, b in list(zip(xs, outs, batches))[:5]:
            assert gb.fft_server_wait(srv, submit(x, y, b), 60.0)["status"] == 0
        assert gb.fft_server_stats(srv)["coalesced_jobs"] == 0
        _check(xs[:5], want[:5], outs[:5])
        gb.fft_server_pause(srv, True)
        tickets = [submit(x, y, b) for x, y, b in zip(xs, outs, batches)]
        gb.fft_server_pause(srv, False)
        assert all(gb.fft_server_wait(srv, k, 60.0)["status"] == 0 for k in tickets)
        assert gb.fft_server_stats(srv)["coalesced_jobs"] == (len(batches) if logn <= 14 else 0)
    finally:
        gb.fft_server_destroy(srv)
    _check(xs, want, outs)


@pytest.mark.parametrize("logn", [15, 17, 18, 20])
def test_server_large(gb, logn):
    """Jobs large enough for fft_execute to join the passes."""
    n, xs, want, outs = _case(gb, logn, [(3 << 22 >> logn) + 1], -1)
    srv = gb.fft_server_create(memory_budget_bytes=4 << 30)
    try:
        k = gb.fft_server_submit(srv, n, xs[0].numel() // n, -1, 0, xs[0].data_ptr(), outs[0].data_ptr())
        assert gb.fft_server_wait(srv, k, 60.0)["status"] == 0
    finally:
        gb.fft_server_destroy(srv)
    _check(xs, want, outs)


@pytest.mark.parametrize("logn", range(0, 24))
@pytest.mark.parametrize("direction", [-1, 1])
def test_noalloc(gb, logn, direction):
    """Every length, the largest batch of the two-pass ones included, in and out of place."""
    t = max(1, 4096 >> logn)
    batches = [1, 3 * t + 1] if logn <= 14 else sorted({1, min(3, 2 ** 23 >> logn), 2 ** 23 >> logn})
    n, xs, want, outs = _case(gb, logn, batches, direction)
    s = torch.cuda.current_stream().cuda_stream
    for x, y, b in zip(xs, outs, batches):
        gb.fft_execute_noalloc(n, b, direction, x.data_ptr(), y.data_ptr(), s)
    _check(xs, want, outs)
    gb.fft_execute_noalloc(n, batches[-1], direction, xs[-1].data_ptr(), xs[-1].data_ptr(), s)
    torch.cuda.synchronize()
    assert torch.equal(_bits(xs[-1]), _bits(want[-1]))


@pytest.mark.parametrize("logn", range(1, 13))
@pytest.mark.parametrize("direction", [-1, 1])
def test_queue(gb, logn, direction):
    """Jobs below, at and above a tile, more tiles than worker blocks, in place."""
    t = max(1, 4096 >> logn)
    batches = [1, t, t + 1, 9 * t - 1]
    n, xs, want, outs = _case(gb, logn, batches, direction)
    for blocks in (0, 2):
        for y in outs:
            y[:-1].zero_()
        torch.cuda.synchronize()
        with gb.Queue(n, max(batches), direction, blocks=blocks) as q:
            for k in [q.submit_ptr(x.data_ptr(), y.data_ptr(), b) for x, y, b in zip(xs, outs, batches)]:
                q.wait(k, 10.0)
        _check(xs, want, outs)
    with gb.Queue(n, max(batches), direction) as q:
        q.wait(q.submit_ptr(xs[-1].data_ptr(), xs[-1].data_ptr(), batches[-1]), 10.0)
    torch.cuda.synchronize()
    assert torch.equal(_bits(xs[-1]), _bits(want[-1]))


@pytest.mark.parametrize("shape,batch", [((8, 8), 700), ((16, 1024), 3), ((64, 64), 33), ((128, 2048), 2),
                                         ((512, 256), 101), ((1024, 512), 25), ((2048, 16), 5), ((4096, 64), 3),
                                         ((32, 16384), 2), ((1, 64), 9), ((64, 1), 9)])
@pytest.mark.parametrize("direction", [-1, 1])
def test_frames(gb, shape, batch, direction):
    """Frames, joined or not: a graph, host buffers, server jobs of the whole batch and of
    parts of it, and another stream beyond those that have counters."""
    torch.manual_seed(batch)
    x = torch.randn((batch,) + shape, dtype=torch.complex64, device="cuda")
    host = x.cpu().pin_memory()
    back, tmp = torch.empty_like(host).pin_memory(), torch.empty_like(x)
    with gb.Plan(shape, batch, direction) as p:
        want = p.execute(x)
        torch.cuda.synchronize()
        outs = [p.execute_graph(x, torch.empty_like(x))]
        streams = [torch.cuda.Stream() for _ in range(5)]
        outs += [p.execute(x, torch.empty_like(x), stream=s) for s in streams]
        torch.cuda.synchronize()
        p.execute_host(host, back, tmp, tmp)
        torch.cuda.synchronize()
    cut = batch // 2
    whole, parts = torch.empty_like(x), torch.empty_like(x)
    torch.cuda.synchronize()
    srv = gb.fft_server_create(memory_budget_bytes=4 << 30)
    try:
        jobs = [(x, whole, batch), (x[:cut], parts[:cut], cut), (x[cut:], parts[cut:], batch - cut)]
        tickets = [gb.fft_server_submit(srv, shape, b, direction, 0, i.data_ptr(), o.data_ptr())
                   for i, o, b in jobs]
        assert all(gb.fft_server_wait(srv, k, 60.0)["status"] == 0 for k in tickets)
    finally:
        gb.fft_server_destroy(srv)
    for y in outs + [back.cuda(), whole, parts]:
        assert torch.equal(_bits(y), _bits(want))


@pytest.mark.parametrize("n,batch", [(2, 2200001), (64, 70001), (1024, 5001), (2048, 2101), (4096, 1051), (16384, 301),
                                     (2 ** 15, 391), (2 ** 18, 49), (2 ** 20, 13), (2 ** 21, 7)])
@pytest.mark.parametrize("direction", [-1, 1])
def test_graph_and_host(gb, n, batch, direction):
    """Graphs, and host buffers in chunks that are a launch each."""
    torch.manual_seed(batch)
    x = torch.randn((batch, n), dtype=torch.complex64, device="cuda")
    host = x.cpu().pin_memory()
    back, tmp = torch.empty_like(host).pin_memory(), torch.empty_like(x)
    with gb.Plan(n, batch, direction) as p:
        want = p.execute(x)
        torch.cuda.synchronize()
        y = p.execute_graph(x, torch.empty_like(x))
        p.execute_host(host, back, tmp, tmp)
        torch.cuda.synchronize()
    assert torch.equal(_bits(y), _bits(want)) and torch.equal(back, want.cpu())
