"""The FP64 path's relativistic recovery (sr_prim_fp64, csrc/sr_df.cuh), compiled
for the host: seeded in double-float, it ends no further from a long double
solution than the float64 iteration (sr_prim64) it stands for, up to Lorentz
factors of a thousand."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1110_0740_gb300", "csrc")


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    exe = str(tmp_path_factory.mktemp("sr") / "sr_fp64")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", os.path.join(HERE, "host"), "-I", CSRC,
                    os.path.join(HERE, "host", "sr_fp64.cpp"), "-o", exe], check=True)
    return exe


# Both amplify float64 roundings by gamma^2 W / p; the bound leaves 1.5 for the
# different roundings of the two forms (10000 states: the mean of a heavy tail).
@pytest.mark.parametrize("lorentz", [1.5, 10, 100, 300, 1000])
def test_no_further_off_than_the_float64_iteration(prog, lorentz):
    out = subprocess.run([prog, str(lorentz), "10000", "3"], check=True, capture_output=True, text=True).stdout
    old_failed, failed, old, err = map(float, out.split())
    assert old_failed == 0 and failed == 0
    assert err <= 1.5 * old
