"""A nan in any variable of one cell raises the step's status, in every dimension,
precision and for the relativistic path too."""
import numpy as np
import pytest

import oracle as O
from paper_1110_0740_gb300 import workloads as W
from tests.gpu_util import gpu_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("recon", [0, 1], ids=["mc", "ppm"])
@pytest.mark.parametrize("ndim", [1, 2, 3])
def test_nan_raises_the_status(ndim, recon, precision):
    n = [9] * ndim + [1] * (3 - ndim)
    for sign in (1.0, -1.0):
        for q in range(9):
            U0 = np.zeros(O.shape(n, ndim))
            rng = np.random.default_rng(q)
            sh = O.interior(U0, n, ndim).shape[1:]
            r = lambda c, s: c + s * (2 * rng.random(sh) - 1)
            V = [r(1, .2), r(.2, .2), r(0, .2), r(0, .2), r(1, .2), r(.5, .2), r(.3, .2), r(0, .2), r(0, .05)]
            O.interior(U0, n, ndim)[:] = W.ideal_cons(V, 5 / 3)
            O.interior(U0, n, ndim)[(q,) + tuple(k // 2 for k in sh)] = np.copysign(np.nan, sign)
            st = gpu_run(U0, n, ndim, [1 / 9] * ndim, 1, 0.3, precision=precision, recon=recon)[2]
            assert st != 0, (q, sign)


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("ndim", [1, 2, 3])
def test_nan_raises_the_relativistic_status(ndim, precision):
    n = [9] * ndim + [1] * (3 - ndim)
    for sign in (1.0, -1.0):
        for q in range(9):
            U0 = np.zeros(O.shape(n, ndim))
            rng = np.random.default_rng(q)
            sh = O.interior(U0, n, ndim).shape[1:]
            r = lambda c, s: c + s * (2 * rng.random(sh) - 1)
            V = [r(1, .2), r(.2, .2), r(0, .2), r(0, .2), r(1, .2), r(.5, .2), r(.3, .2), r(0, .2), r(0, .05)]
            O.interior(U0, n, ndim)[:] = W.srmhd_cons(V, 4 / 3)
            O.interior(U0, n, ndim)[(q,) + tuple(k // 2 for k in sh)] = np.copysign(np.nan, sign)
            st = gpu_run(U0, n, ndim, [1 / 9] * ndim, 1, 0.3, precision=precision, gamma=4 / 3, physics=1)[2]
            assert st != 0, (q, sign)
