"""The Python binding without torch: plans are made and run from pointers by programs
that have no torch, so only calls that take tensors may import it."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import sys
sys.modules["torch"] = None  # `import torch` raises ImportError
from paper_1505_08067_gb300 import gbfft

class Fake:  # the C library: every call succeeds
    def __getattr__(self, name):
        return lambda *a: 0

gbfft.load = lambda: Fake()
p = gbfft.Plan((4, 8), 3, gbfft.FFT_INVERSE, gbfft.FFT_PREC_FP32)
assert p.elements == 96 and not hasattr(p, "nothing")
class Buffer:
    def data_ptr(self):
        return 16
p.execute_host(Buffer(), Buffer(), Buffer(), Buffer(), stream=0)
gbfft.fft_execute(p.handle, 16, 32, 0)
p.close()
"""


def test_plan_without_torch():
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr


def test_first_execute_finds_the_type(monkeypatch):
    """Where torch is loaded, a plan is complete: its first execute looks nothing up, and
    no attribute of any execute goes through a hook of the class."""
    torch = pytest.importorskip("torch")
    from paper_1505_08067_gb300 import gbfft

    class Fake:
        def __getattr__(self, name):
            return lambda *a: 0

    monkeypatch.setattr(gbfft, "load", lambda: Fake())
    for precision, dtype in ((gbfft.FFT_PREC_FP32, torch.complex64), (gbfft.FFT_PREC_TC_FP16_C32, torch.complex32)):
        p = gbfft.Plan(8, 3, gbfft.FFT_FORWARD, precision)
        assert p.__dict__["_dtype"] is dtype
        p.close()
    assert not hasattr(gbfft.Plan, "__getattr__")
