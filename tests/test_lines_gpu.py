"""The short-line kernels (contiguous transforms of 2^3 .. 2^10 points, fast
convolution of lines and columns of 2^3 .. 2^11) at the edges of their tiles: one
line, one short of a tile, a tile, one more, many; 8-byte aligned buffers, in
place, through the chunked host path, against the oracle."""
import numpy as np
import pytest

from paper_1505_08067_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("logn", range(3, 11))
@pytest.mark.parametrize("direction", [-1, 1])
def test_lines(gb, oracle, logn, direction):
    n = 2 ** logn
    tile = 4096 // n
    for batch in (1, tile - 1, tile, tile + 1, 37 * tile + 3):
        x_np = synth.uniform(900 + logn, batch, n)
        buf = torch.empty(batch * n + 1, dtype=torch.complex64, device="cuda")
        guard = torch.full((batch * n + 2,), 7.0 + 7.0j, dtype=torch.complex64, device="cuda")
        with gb.Plan(n, batch, direction) as p:
            assert p.describe()["kernels"][0]["lines"] == 1
            first = None
            for shift in (0, 1):
                x = buf[shift:shift + batch * n]
                x.copy_(torch.from_numpy(x_np).view(-1))
                y = guard[shift:shift + batch * n]
                p.execute(x, y)
                assert torch.all(guard[shift + batch * n:] == 7.0 + 7.0j)  # nothing past the last line
                first = y.clone() if first is None else first
                assert torch.equal(first, y)
            p.execute(x, x)
            assert torch.equal(first, x)
        err = oracle.rel_l2(first.view(batch, n).cpu().numpy(), oracle.fft(x_np, direction))
        assert np.max(err) <= 1e-6 * max(1.0, logn), batch


def test_lines_host_chunks(gb):
    """fft_execute_host in several chunks of about 32 MiB, the last one short."""
    n, batch = 64, 150001
    x = torch.from_numpy(synth.uniform(931, batch, n)).pin_memory()
    y = torch.empty_like(x).pin_memory()
    d, e = torch.empty(x.shape, dtype=x.dtype, device="cuda"), torch.empty(x.shape, dtype=x.dtype, device="cuda")
    with gb.Plan(n, batch) as p:
        p.execute_host(x, y, d, e)
        torch.cuda.synchronize()
        assert torch.equal(y, p.execute(x.cuda()).cpu())


@pytest.mark.parametrize("logn", range(3, 12))
@pytest.mark.parametrize("per_line", [False, True])
def test_conv_lines(gb, oracle, logn, per_line):
    n = 2 ** logn
    tile = max(1, 4096 // n)
    for batch in (1, tile + 1, 5 * tile - 1):
        lines = batch if per_line else 1
        x_np, h_np = synth.uniform(940 + logn, batch, n), synth.uniform(960 + logn, lines, n)
        h = torch.from_numpy(h_np).cuda()
        x = torch.from_numpy(x_np).cuda()
        with gb.ConvPlan(n, batch, [(h, lines, 1.0 / n)]) as p:
            assert p.describe()["kernels"][0]["lines"] == 1
            y = p.execute(x)
            p.execute(x, x)
            assert torch.equal(x, y)
        ref = np.fft.ifft(np.fft.fft(x_np.astype(np.complex128)) * h_np)
        assert np.max(oracle.rel_l2(y.cpu().numpy(), ref)) <= 2e-6 * logn, batch


@pytest.mark.parametrize("rows,cols,batch", [(8, 2048, 3), (32, 4, 70), (128, 64, 1), (512, 8, 5),
                                             (1024, 32, 2), (2048, 16, 3)])
@pytest.mark.parametrize("per_line", [(False, False), (True, True), (True, False)])
def test_conv_columns(gb, oracle, rows, cols, batch, per_line):
    """Frames of fewer columns than a tile, and of more; one filter per column,
    per row, or shared."""
    x_np = synth.uniform(981, batch, rows * cols).reshape(batch, rows, cols)
    hc = synth.uniform(982, rows, cols if per_line[0] else 1)
    hr = synth.uniform(983, rows if per_line[1] else 1, cols)
    x = torch.from_numpy(x_np).cuda()
    with gb.ConvPlan((rows, cols), batch, [(torch.from_numpy(hc).cuda(), hc.shape[1], 1.0 / rows),
                                           (torch.from_numpy(hr).cuda(), hr.shape[0], 1.0 / cols)]) as p:
        assert p.describe()["kernels"][1]["lines"] == 1
        y = p.execute(x)
        torch.cuda.synchronize()
    ref = np.fft.ifft(np.fft.fft(x_np.astype(np.complex128)) * hr[None])
    ref = np.fft.ifft(np.fft.fft(ref, axis=1) * hc[None], axis=1)
    err = oracle.rel_l2(y.cpu().numpy().reshape(batch, -1), ref.reshape(batch, -1))
    assert np.max(err) <= 2e-6 * np.log2(rows * cols)


def test_conv_host_chunks(gb, oracle):
    """Per-line filters through fft_execute_host: each chunk starts at its own
    line's filter."""
    n, batch = 512, 20001
    x_np, h_np = synth.uniform(990, batch, n), synth.uniform(991, batch, n)
    x, y = torch.from_numpy(x_np).pin_memory(), torch.empty(batch, n, dtype=torch.complex64).pin_memory()
    d, e = torch.empty(batch, n, dtype=torch.complex64, device="cuda"), torch.empty(batch, n, dtype=torch.complex64, device="cuda")
    with gb.ConvPlan(n, batch, [(torch.from_numpy(h_np).cuda(), batch, 1.0 / n)]) as p:
        p.execute_host(x, y, d, e)
        torch.cuda.synchronize()
        assert torch.equal(y, p.execute(x.cuda()).cpu())
    idx = np.array([0, 8191, 8192, 16384, 20000])
    ref = np.fft.ifft(np.fft.fft(x_np[idx].astype(np.complex128)) * h_np[idx])
    assert np.max(oracle.rel_l2(y.numpy()[idx], ref)) <= 2e-6 * 9
