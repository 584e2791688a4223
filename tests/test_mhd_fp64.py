"""The FP64 path's forms of the ideal-MHD arithmetic (csrc/mhd_fp64.cuh), compiled
for the host beside the generic functions they stand for."""
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
    exe = str(tmp_path_factory.mktemp("mhd") / "mhd_fp64")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", os.path.join(HERE, "host"), "-I", CSRC,
                    os.path.join(HERE, "host", "mhd_fp64.cpp"), "-o", exe], check=True)
    return exe


def test_a_nan_stays_one(prog):
    """No flux and no predicted value is a number where the generic functions,
    whose comparisons a nan fails, give a nan."""
    lost, both = map(int, subprocess.run([prog, "nan"], check=True, capture_output=True, text=True).stdout.split())
    assert both > 100000
    assert lost == 0


def test_no_less_accurate_than_ieee_forms(prog):
    """Against long double, on 200000 random states from nearly uniform to rough:
    the predicted states (MC, PPM) and the HLLD fluxes are no further off than the
    generic functions' in IEEE double."""
    out = subprocess.run([prog, "err", "200000", "1"], check=True, capture_output=True, text=True).stdout
    for ieee, here in (map(float, line.split()) for line in out.splitlines()):
        assert 0.0 < here <= ieee
