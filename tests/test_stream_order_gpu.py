"""Launches that may start while the kernel before them finishes: chains of
dependent executions, each reading what the last one wrote and overwriting what
it read, without any synchronisation, give bit for bit what the same chain gives
with one after every step -- every kernel family, next to each other and next to
other kernels, copies and fills of the stream, and replayed from a graph."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (shape, precision, options): 2^17 elements each
PLANS = [((8, ), 0, {}), ((64,), 0, {}), ((1024,), 0, {}), ((1024,), 0, {"variant": 1}), ((4096,), 0, {}),
         ((4096,), 0, {"variant": 3}), ((8192,), 0, {}), ((16384,), 0, {}), ((16,), 0, {"generic": 1}),
         ((2 ** 16,), 0, {}), ((2 ** 17,), 0, {"variant": 2}), ((64, 64), 0, {}), ((4096, 32), 0, {}),
         ((32, 4096), 0, {"variant": 1}), ((4096,), 3, {}), ((16384,), 1, {}), ((4096,), 2, {"variant": 1}),
         ((2 ** 16,), 3, {}), ((2 ** 17,), 1, {})]
E = 2 ** 17


def _chain(plans, x, y, sync, stream):
    a, b = x, y
    for rep in range(6):
        for p in plans:
            p(a, b)                     # b <- P(a)
            if sync:
                torch.cuda.synchronize()
            b.mul_(0.004)               # a torch kernel between two of ours
            if sync:
                torch.cuda.synchronize()
            a, b = b, a
        plans[rep % len(plans)](a, a)   # in place, right after the last
        if sync:
            torch.cuda.synchronize()
        a.mul_(0.004)
    return a.clone()


def test_chain(gb):
    made = []
    for i, (shape, prec, opts) in enumerate(PLANS):
        n = 1
        for v in shape:
            n *= v
        made.append(gb.Plan(shape if len(shape) > 1 else shape[0], E // n, 1 if i % 2 else -1, prec, **opts))
    h = torch.randn(512, dtype=torch.complex64, device="cuda")
    made.append(gb.ConvPlan(512, E // 512, [(h, 1, 1.0 / 512)]))
    hc = torch.randn(32, 1, dtype=torch.complex64, device="cuda")
    made.append(gb.ConvPlan((32, 512), E // (32 * 512), [(hc, 1, 1.0 / 32), (h, 1, 1.0 / 512)]))
    stream = torch.cuda.Stream()
    runs = [lambda a, b, p=p: gb.fft_execute(p.handle, a.data_ptr(), b.data_ptr(), stream.cuda_stream) for p in made]
    torch.manual_seed(5)
    x0 = torch.randn(E, dtype=torch.complex64, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        want = _chain(runs, x0.clone(), torch.zeros_like(x0), True, stream)
        for _ in range(5):
            got = _chain(runs, x0.clone(), torch.zeros_like(x0), False, stream)
            torch.cuda.synchronize()
            assert torch.isfinite(torch.view_as_real(got)).all() and torch.equal(got, want)
    # our kernels back to back, without anything between them
    def straight(sync):
        a, b = x0.clone(), torch.zeros_like(x0)
        for r in runs:
            r(a, b)
            if sync:
                torch.cuda.synchronize()
            r(b, a)
            if sync:
                torch.cuda.synchronize()
            a.mul_(1e-3)
        return a.clone()
    with torch.cuda.stream(stream):
        want = straight(True)
        for _ in range(10):
            got = straight(False)
            torch.cuda.synchronize()
            assert torch.equal(got.view(torch.int64), want.view(torch.int64))  # bits: it may overflow
    for p in made:
        p.close()


def test_chain_in_graph(gb):
    """The same dependence inside a graph the caller captures."""
    n, batch = 1024, 64
    with gb.Plan(n, batch, -1) as p, gb.Plan(n, batch, 1) as q, gb.Plan(2 ** 16, 1, -1) as r:
        x = torch.randn(n * batch, dtype=torch.complex64, device="cuda")
        y, z = torch.empty_like(x), torch.empty_like(x)
        s = torch.cuda.Stream()
        torch.cuda.synchronize()

        def work():
            for _ in range(4):
                gb.fft_execute(p.handle, x.data_ptr(), y.data_ptr(), s.cuda_stream)
                gb.fft_execute(r.handle, y.data_ptr(), z.data_ptr(), s.cuda_stream)
                gb.fft_execute(q.handle, z.data_ptr(), y.data_ptr(), s.cuda_stream)
        with torch.cuda.stream(s):
            work()
            torch.cuda.synchronize()
            want = y.clone()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                work()
            for _ in range(10):
                y.zero_()
                g.replay()
                torch.cuda.synchronize()
                assert torch.equal(y, want)
