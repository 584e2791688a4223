"""Relativistic steps in other units: a state scaled by a power of two (rho, p, m,
E by 4^k, B and psi by 2^k) steps to the scaled result, for both equations of
state, in the mixed and the FP64 path."""
import numpy as np
import pytest

import oracle as O
from tests.gpu_util import gpu_run
from tests.test_gpu_srmhd_sweeps import _state

pytestmark = pytest.mark.gpu


# Scaling by powers of two moves no rounding, except where a float32 product of
# slopes underflows (slopes below 2^-63): one float32 rounding (6e-8) in a few cells of
# ten thousand, 1e-9 in the mean square; float64 has none
@pytest.mark.parametrize("precision,tol", [(0, 1e-14), (1, 1e-9)], ids=["fp64", "mixed"])
@pytest.mark.parametrize("tm", [0, 1], ids=["ideal", "taub-mathews"])
@pytest.mark.parametrize("k", [-20, -12, 12])
def test_a_scaled_state_steps_alike(precision, tol, tm, k):
    n, gamma = [21, 18, 20], 0.0 if tm else 4.0 / 3.0
    U0 = _state(n, 3, (0, 1, 2), gamma)
    s = np.array([4.0 ** k] * 5 + [2.0 ** k] * 4).reshape(9, 1, 1, 1)
    out = []
    for U in (U0, U0 * s):
        got, dts, st = gpu_run(U, n, 3, [1 / 21] * 3, 2, 0.3, precision=precision, gamma=gamma, physics=1, eos=tm)
        assert st == 0
        out.append((O.interior(got, n, 3), dts))
    (a, da), (b, db) = out
    b = b / s
    assert np.allclose(da, db, rtol=tol, atol=0.0)
    for q in range(9):
        assert np.linalg.norm(a[q] - b[q]) <= tol * max(np.linalg.norm(a[q]), np.linalg.norm(a[5:8])), q
