"""The FP64 path's reciprocal and roots (csrc/mhd_fp64.cuh) on the device, over the
whole exponent range."""
import os
import subprocess

import pytest

from paper_1110_0740_gb300 import _build

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_reciprocal_and_roots(tmp_path):
    """In units of 2^-53 relative, from seeds good to 2^-22: 1/x rounds once (1, and
    2^-16 from the cube of the seed's error); 1/sqrt(x) adds half the rounding of x y
    (1.5); sqrt(x) half of it once more (2)."""
    exe = str(tmp_path / "roots")
    subprocess.run([_build.nvcc(), *_build.flags(), os.path.join(HERE, "device", "fp64_roots.cu"), "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    rcp, rsqrt, sqrt = map(float, out[:3])
    assert rcp <= 1.01 and rsqrt <= 1.51 and sqrt <= 2.01
    assert out[3:] == ["0", "0", "0", "0"]
