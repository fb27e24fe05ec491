"""The work that the library's users give it, as cases that a program can prepare, run and check.

Three kinds of plan, each through ``gbfft.Plan`` / ``gbfft.ConvPlan`` with the
library's own choice of kernels (no options), on data that is on the GPU:

* ``lines``: a batch of 1D transforms of one length;
* ``frames``: a batch of 2D frames (a row pass, then a column pass);
* ``compress``: fast convolution of lines or frames with matched filters.

A case names the kind, ``rows`` (frames and 2D compression; 0 for lines),
``cols`` (the length of a line), ``batch``, ``inverse``, ``prec`` (``fp32``, or a
tensor-core class: ``fp16``, ``bf16``, ``bf16x3``, ``c32`` for FP16 with complex32
data) and, for compression, which dimensions have one filter per line
(``per_row``, ``per_col``) rather than one shared filter.
"""
import math

import torch

from paper_1505_08067_gb300 import gbfft

_PREC = {"fp32": gbfft.FFT_PREC_FP32, "fp16": gbfft.FFT_PREC_TC_FP16, "bf16": gbfft.FFT_PREC_TC_BF16,
         "bf16x3": gbfft.FFT_PREC_TC_BF16X3, "c32": gbfft.FFT_PREC_TC_FP16_C32}


def _lines(n, batch, inverse=False, prec="fp32"):
    return {"kind": "lines", "rows": 0, "cols": n, "batch": batch, "inverse": inverse, "prec": prec,
            "per_row": False, "per_col": False}


def _frames(rows, cols, batch, inverse=False):
    return {"kind": "frames", "rows": rows, "cols": cols, "batch": batch, "inverse": inverse,
            "prec": "fp32", "per_row": False, "per_col": False}


def _compress(rows, cols, batch, per_row=False, per_col=False):
    return {"kind": "compress", "rows": rows, "cols": cols, "batch": batch, "inverse": False,
            "prec": "fp32", "per_row": per_row, "per_col": per_col}


def listed():
    return [
        # one call on a small batch, as a real-time loop makes it: latency
        dict(_lines(1024, 64), name="call-1024x64"),
        # pulse-Doppler processing: many short lines, a count that fills no tile evenly
        dict(_lines(64, 100003), name="lines-64x100003"),
        # an ordinary batch of lines, about one L2 in and out
        dict(_lines(4096, 3001), name="lines-4096x3001"),
        # the longest on-chip transform at the batched sweep's size, backward
        dict(_lines(16384, 8192, True), name="lines-16384x8192-inv"),
        # middle lengths of the two-pass path (a spectrogram's long windows), odd batch
        dict(_lines(1 << 17, 75), name="lines-2^17x75"),
        # one long record on its own, backward: latency of the two-pass path
        dict(_lines(1 << 20, 1, True), name="lines-2^20x1-inv"),
        # the two-pass path's throughput
        dict(_lines(1 << 22, 16), name="lines-2^22x16"),
        # one SAR frame: range FFTs, then azimuth FFTs
        dict(_frames(4096, 8192, 1), name="sar-frame-4096x8192"),
        # a stack of smaller frames or images, backward
        dict(_frames(1024, 512, 25, True), name="frames-1024x512x25-inv"),
        # range and azimuth compression of one raw SAR frame: one range replica,
        # one azimuth filter per range bin
        dict(_compress(4096, 8192, 1, per_col=True), name="sar-compress-4096x8192"),
        # the tensor-core class with half the bytes per element
        dict(_lines(8192, 8192, False, "c32"), name="tc-c32-8192x8192"),
        # the compensated tensor-core class above one on-chip block
        dict(_lines(1 << 20, 16, False, "bf16x3"), name="tc-bf16x3-2^20x16"),
    ]


def _loguniform(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    # elements: from a few thousand to 2^26 (2^25 where each costs more than
    # one pass over memory), below the largest listed case
    kind = rng.choice(["lines", "lines", "lines", "frames", "frames", "tc", "tc", "compress"])
    elems = _loguniform(rng, 1 << 12, 1 << 25)
    if kind == "lines":
        n = 1 << rng.randint(4, 24)
        if n <= 1 << 14:
            elems = min(1 << 26, elems * 2)
        return _lines(n, max(1, elems // n), rng.random() < 0.5)
    if kind == "tc":
        n = 1 << rng.randint(6, 22)
        prec = rng.choice(["fp16", "bf16", "bf16x3", "c32"])
        return _lines(n, max(1, elems // n), rng.random() < 0.5, prec)
    if kind == "frames":
        rows, cols = 1 << rng.randint(4, 13), 1 << rng.randint(4, 13)
        if rows * cols > 1 << 25:
            rows = (1 << 25) // cols
        return _frames(rows, cols, max(1, elems // (rows * cols)), rng.random() < 0.5)
    rows, cols = rng.choice([0, 1 << rng.randint(5, 12)]), 1 << rng.randint(5, 13)
    return _compress(rows, cols, max(1, elems // (max(1, rows) * cols)), rng.random() < 0.5,
                     rows > 0 and rng.random() < 0.5)


def _shape(case):
    return (case["batch"],) + ((case["rows"],) if case["rows"] else ()) + (case["cols"],)


def _chirp(n, width, rate, device="cuda"):
    """A linear-FM pulse of `width` samples (its rate in cycles per sample^2) in n samples, FP64."""
    t = torch.arange(width, dtype=torch.float64, device=device) - (width - 1) / 2
    s = torch.zeros(n, dtype=torch.complex128, device=device)
    s[:width] = torch.polar(torch.ones_like(t), math.pi * rate * t * t)
    return s


def _azimuth_rate(cols, rows):
    """The azimuth chirp's rate in each range bin: it falls across the swath."""
    width = max(2, rows // 8)
    c = torch.arange(cols, dtype=torch.float64, device="cuda") / cols
    return width, 0.8 / (width * (1 + c / 2))


def _input(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    shape = _shape(case)
    if case["rows"] >= 512 and case["cols"] >= 512:
        # a radar frame: echoes of point scatterers in receiver noise
        x = torch.view_as_complex(torch.randn(shape + (2,), generator=g, device="cuda")).mul_(0.22)
        rows, cols = case["rows"], case["cols"]
        rng = _chirp(cols, cols // 16, 0.8 * 16 / cols)[:cols // 16].to(torch.complex64)
        width, rates = _azimuth_rate(cols, rows)
        at = torch.rand(24, 3, generator=g, device="cuda").tolist()
        for u, v, phase in at:
            r, c = int(u * (rows - width)), int(v * (cols - rng.numel()))
            az = _chirp(width, width, float(rates[c])).to(torch.complex64) * complex(math.cos(6.28 * phase), math.sin(6.28 * phase))
            x[:, r:r + width, c:c + rng.numel()] += az[:, None] * rng[None, :]
    else:
        # noise in the receiver's range, parts uniform in [-1, 1)
        x = torch.view_as_complex(torch.rand(shape + (2,), generator=g, device="cuda").mul_(2).sub_(1))
    if case["prec"] == "c32":
        x = torch.view_as_complex(torch.view_as_real(x).half())
    return x


def _filters(case):
    """The matched filters' spectra per dimension (FP32, as a program keeps them): [(h, lines, scale)]."""
    rows, cols = case["rows"], case["cols"]
    replica = _chirp(cols, max(2, cols // 16), 0.8 * 16 / cols)
    hr = torch.fft.fft(replica).conj()
    lines = rows if rows else case["batch"]
    if case["per_row"]:  # a replica of its own phase for each line
        turn = torch.arange(lines, dtype=torch.float64, device="cuda")
        row = torch.polar(torch.ones_like(turn), turn)[:, None].to(torch.complex64) * hr.to(torch.complex64)
    else:
        row = hr.to(torch.complex64)
    row = (row.contiguous(), lines if case["per_row"] else 1, 1.0 / cols)
    if not rows:
        return [row]
    width, rates = _azimuth_rate(cols, rows)
    if not case["per_col"]:
        rates = rates[:1]
    t = torch.arange(width, dtype=torch.float64, device="cuda") - (width - 1) / 2
    az = torch.zeros(rows, rates.numel(), dtype=torch.complex64, device="cuda")
    az[:width] = torch.polar(torch.ones((), dtype=torch.float64, device="cuda").expand(width, rates.numel()),
                             math.pi * rates[None, :] * t[:, None] * t[:, None]).to(torch.complex64)
    col = torch.fft.fft(az, dim=0).conj().resolve_conj().contiguous()
    return [(col, cols if case["per_col"] else 1, 1.0 / rows), row]


def prepare(case, seed):
    n = (case["rows"], case["cols"]) if case["rows"] else case["cols"]
    x = _input(case, seed)
    if case["kind"] == "compress":
        plan = gbfft.ConvPlan(n, case["batch"], _filters(case))
    else:
        plan = gbfft.Plan(n, case["batch"], gbfft.FFT_INVERSE if case["inverse"] else gbfft.FFT_FORWARD,
                          _PREC[case["prec"]])
    return {"plan": plan, "x": x, "out": torch.empty_like(x)}


def run(state):
    return state["plan"].execute(state["x"], state["out"])


def work(case):
    elems = math.prod(_shape(case))
    per = max(1, case["rows"]) * case["cols"]
    size = 4 if case["prec"] == "c32" else 8
    nbytes, flops = 2 * size * elems, 5.0 * elems * math.log2(per)
    if case["kind"] == "compress":
        lines = case["rows"] or case["batch"]
        nbytes += 8 * case["cols"] * (lines if case["per_row"] else 1)
        nbytes += 8 * case["rows"] * (case["cols"] if case["per_col"] else 1)
        flops = 2 * flops + 6.0 * elems * (2 if case["rows"] else 1)
    return {"bytes": nbytes, "flops": flops}


def exact(case, seed):
    x = _input(case, seed)
    if case["prec"] == "c32":
        x = torch.view_as_complex(torch.view_as_real(x).double())
    else:
        x = x.to(torch.complex128)
    if case["kind"] == "compress":
        dims = [-1] if not case["rows"] else [-1, -2]
        filters = _filters(case)[::-1]
        for dim, (h, lines, scale) in zip(dims, filters):
            h = h.to(torch.complex128)
            if dim == -2:  # one column filter per range bin, or one for all
                h = h.reshape(case["rows"], lines)
            elif lines > 1:
                h = h.reshape(((case["rows"] or case["batch"]), case["cols"]))
            n = x.shape[dim]
            f = torch.fft.fft(x, dim=dim)
            f *= h
            x = torch.fft.ifft(f, dim=dim)
            x *= n * scale
            del f
        return x
    dims = (-2, -1) if case["rows"] else (-1,)
    if case["inverse"]:
        return torch.fft.ifftn(x, dim=dims, norm="forward")
    return torch.fft.fftn(x, dim=dims)
