"""The mixed relativistic recoveries on the device (csrc/sr_df.cuh, compiled as the
library compiles them): wherever the double-float ones decide, the float64
iterations' results rounded to float32, bit for bit, in any units."""
import os
import subprocess

import pytest

from paper_1110_0740_gb300 import _build

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("sr") / "sr_recover")
    subprocess.run([_build.nvcc(), *_build.SOURCE_FLAGS["ctu_sr32.cu"], *_build.flags(),
                    os.path.join(HERE, "device", "sr_recover.cu"), "-o", exe], check=True)
    return exe


# decided: nearly all with tau in [2^-16, 2^16), none far outside (tests/test_sr_scale.py)
@pytest.mark.parametrize("k", [-40, -16, -12, -10, -9, -8, -7, -4, 0, 1, 5, 12, 40])
def test_double_float_is_the_float64_iteration(prog, k):
    out = subprocess.run([prog, str(k), "1000000"], check=True, capture_output=True, text=True).stdout
    physical, wrong, decided = map(int, out.split())
    assert physical > 900000
    assert wrong == 0
    if k in (-4, 0, 1):
        assert decided >= 0.95 * physical
