"""The double-float relativistic recovery (csrc/sr_df.cuh), compiled for the
host: wherever it decides, rho, v and p are the float64 iteration's rounded to
float32, bit for bit, and it leaves few physical states undecided."""
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
    exe = str(tmp_path_factory.mktemp("sr") / "sr_recover")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", os.path.join(HERE, "host"), "-I", CSRC,
                    os.path.join(HERE, "host", "sr_recover.cpp"), "-o", exe], check=True)
    return exe


# undecided: the share of values within the certificate's margin (K = 3 units of
# 2^-48, amplified by gamma^2 W / p) of a float32 rounding boundary; 2 % covers
# the beam's edge, where it is largest
@pytest.mark.parametrize("family", [0, 1, 2, 3], ids=["beam", "edge", "ambient", "any"])
def test_recovery_is_the_float64_iterations(prog, family):
    out = subprocess.run([prog, str(family), "200000", "7"], check=True, capture_output=True, text=True).stdout
    physical, undecided, wrong, fwrong = map(int, out.split())
    assert physical > 100000
    assert wrong == 0 and fwrong == 0
    assert undecided <= 0.02 * physical
