"""The relativistic recoveries (csrc/srmhd_device.cuh, csrc/sr_df.cuh), compiled
for the host, in any units: the state scaled by a power of two gives the same
primitives, scaled, bit for bit."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1110_0740_gb300", "csrc")


def build(tmp_path_factory, name, *link, flags=()):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    exe = str(tmp_path_factory.mktemp("sr") / name)
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", *flags, "-I", os.path.join(HERE, "host"), "-I", CSRC, "-c",
                    os.path.join(HERE, "host", name + ".cpp"), "-o", exe + ".o"], check=True)
    subprocess.run([cxx, *link, exe + ".o", "-o", exe], check=True)
    return exe


@pytest.fixture(scope="module")
def prog(tmp_path_factory):
    return build(tmp_path_factory, "sr_scale")


# exponents of two of B: density and pressure from 4^-250 to 4^250
@pytest.mark.parametrize("k", [-250, -100, -40, -20, -10, -7, -3, 3, 7, 20, 40, 250])
def test_float64_recoveries_scale(prog, k):
    out = subprocess.run([prog, str(k), "4000", "5"], check=True, capture_output=True, text=True).stdout
    assert out.split() == ["0", "0"]


@pytest.fixture(scope="module")
def units(tmp_path_factory):
    # -ffast-math at the link alone: the start-up code that flushes denormals
    return build(tmp_path_factory, "sr_units", "-ffast-math", flags=["-DSEED_ULPS=2"])


# undecided: as in test_sr_recover.py (2 %) while 2^-16 <= tau < 2^16 (the states at
# unit scale have 2^-4 < tau < 2^14), all of them far outside
@pytest.mark.parametrize("k", [-55, -30, -20, -16, -13, -12, -11, -10, -9, -8, -7, -6, -4, -2, 0, 1, 2, 3, 4, 5, 6, 7, 9, 12, 45])
def test_double_float_recovery_in_any_units(units, k):
    out = subprocess.run([units, str(k), "100000", "9"], check=True, capture_output=True, text=True).stdout
    flushed, physical, undecided, wrong = map(int, out.split())
    assert flushed == 1 and physical > 90000
    assert wrong == 0
    assert undecided <= (0.02 if -6 <= k <= 1 else 1.0) * physical
