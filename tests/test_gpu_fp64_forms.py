"""The FP64 path's own arithmetic (csrc/mhd_fp64.cuh, sr_prim_fp64) on the
states where its forms branch or degenerate, against the oracle: relative L1
and elementwise within 1e-11 of the largest value, the FP64 bar."""
import numpy as np
import pytest

import oracle as O
from paper_1110_0740_gb300 import workloads as W
from tests.gpu_util import gpu_run

pytestmark = pytest.mark.gpu

N = [11, 9, 10]
DX = [1 / 16] * 3


def _mhd(kind):
    rng = np.random.default_rng(11)
    sh = (N[2], N[1], N[0])
    r = lambda s: s * (2 * rng.random(sh) - 1)
    o = np.ones(sh)
    rho, p, v, B, psi = o + r(.3), o + r(.3), [r(.3) for _ in range(3)], [r(.5) for _ in range(3)], r(.05)
    if kind == "hydro":             # no field: B_t = B_n = 0, psi = 0
        B, psi = [0 * o] * 3, 0 * o
    elif kind == "along_x":         # B_t = 0 for the sweep along x, B_n = 0 for the others
        B, psi = [0.7 * o, 0 * o, 0 * o], 0 * o
    elif kind == "triple":          # a = c_a with B_t = 0: fast, slow and Alfven speeds coincide along x
        rho, p, v, B, psi = o, 0.6 * o, [r(1e-3) for _ in range(3)], [o, 0 * o, 0 * o], 0 * o
    elif kind == "weak":            # B_t around and below the degenerate threshold
        B = [r(.5), r(1e-11), r(1e-13)]
    elif kind == "supersonic":      # every Riemann fan on one side of the face, both signs
        v = [20 * o + r(.3), -20 * o + r(.3), 20 * o + r(.3)]
    elif kind == "uniform":
        rho, p, v, B, psi = o, o, [.1 * o, .2 * o, .3 * o], [.4 * o, .5 * o, .6 * o], 0 * o
    return W.pad_periodic(W.ideal_cons([rho, *v, p, *B, psi], 5 / 3), 3)


@pytest.mark.parametrize("recon", [0, 1], ids=["mc", "ppm"])
@pytest.mark.parametrize("kind", ["random", "hydro", "along_x", "triple", "weak", "supersonic", "uniform"])
def test_mhd_forms(kind, recon):
    U0 = _mhd(kind)
    got, dts, st = gpu_run(U0, N, 3, DX, 2, 0.3, precision=0, recon=recon)
    assert st == 0
    ref = U0.copy()
    for dt, ch in dts:
        ref, bad = O.mhd_step(ref, N, 3, DX, dt, ch, recon=recon)
        assert bad == 0
        O.fill_periodic(ref, N, 3)
    G, R = O.interior(got, N, 3), O.interior(ref, N, 3)
    scale = np.abs(R).max(axis=(1, 2, 3))
    scale[1:4] = max(scale[1:4].max(), 1e-300)  # a component that vanishes is held to its vector
    scale[5:8] = max(scale[5:8].max(), scale[0] * 1e-3)
    scale[8] = max(scale[8], ch * scale[5])
    assert (np.abs(G - R).max(axis=(1, 2, 3)) / scale).max() < 1e-11


@pytest.mark.parametrize("kind", ["beam", "rest", "unmagnetised", "hot"])
def test_relativistic_forms(kind):
    rng = np.random.default_rng(5)
    sh = (N[2], N[1], N[0])
    r = lambda s: s * (2 * rng.random(sh) - 1)
    o = np.ones(sh)
    rho, p, v, B = o + r(.2), .1 * o + r(.02), [r(.02), r(.02), .99 * o + r(.001)], [r(.1), r(.1), 2 * o + r(.1)]
    if kind == "rest":
        v = [0 * o] * 3
    elif kind == "unmagnetised":
        v, B = [r(.3), r(.3), r(.3)], [0 * o] * 3
    elif kind == "hot":
        p, v = 500 * o + r(50), [r(.4), r(.4), r(.4)]
    U0 = W.pad_periodic(W.srmhd_cons([rho, *v, p, *B, 0 * o], 4 / 3), 3)
    got, dts, st = gpu_run(U0, N, 3, DX, 1, 0.2, precision=0, gamma=4 / 3, physics=1)
    assert st == 0
    ref, bad = O.srmhd_step(U0, N, 3, DX, *dts[0], gamma=4 / 3)
    assert bad == 0
    G, R = O.interior(got, N, 3), O.interior(ref, N, 3)
    scale = np.abs(R).max(axis=(1, 2, 3))
    scale[1:4] = max(scale[1:4].max(), scale[0])
    scale[5:8] = max(scale[5:8].max(), scale[0])
    scale[8] = max(scale[8], scale[5])
    assert (np.abs(G - R).max(axis=(1, 2, 3)) / scale).max() < 1e-11
