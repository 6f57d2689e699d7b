"""The fused AdamW epilogues' square root and quotient against the correctly rounded ones."""
import ctypes
import os
import subprocess

import pytest

from tests._gpu import need_gpu

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_sqrt_and_quotient_are_correctly_rounded(tmp_path):
    """sqrt over every significand at exponents of either parity and every subnormal; quotients
    next to a midpoint (the hardest to round), over the whole exponent range, of numerators or
    results too small for a residual (two ulps), and with zeros, infinities and NaN."""
    need_gpu()
    from paper_2406_14898_gb300 import build
    so = str(tmp_path / "arith_check.so")
    subprocess.run([build._nvcc()] + build.NVCC_FLAGS + ["-shared", os.path.join(HERE, "arith_check.cu"), "-o", so],
                   check=True, capture_output=True)
    bad = (ctypes.c_ulonglong * 7)()
    assert ctypes.CDLL(so).arith_check(bad, 7) == 0
    assert list(bad) == [0] * 7
