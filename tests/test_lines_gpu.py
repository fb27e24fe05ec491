"""The short-line kernel (contiguous transforms of 2^3 .. 2^10 points) at the edges
of its tiles: one line, one short of a tile, a tile, one more, many; 8-byte
aligned buffers, in place, through the chunked host path, against the oracle."""
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
