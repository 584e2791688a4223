"""The mixed relativistic sweeps along x, y and z, each with its own float32
predictor and fluxes (csrc/sr_df.cuh), against the oracle: the same state with
its axes permuted, on ragged boxes, in two and three dimensions and for both
equations of state."""
import numpy as np
import pytest

import oracle as O
from paper_1110_0740_gb300 import workloads as W
from tests.gpu_util import gpu_run, maxrel

pytestmark = pytest.mark.gpu

# One step at Lorentz factor up to 3: float32 rounding (2^-24) of the states,
# amplified by gamma^2 W / p ~ 9 x 10 in the recovered pressure and summed over
# the four states behind a flux, gives 2e-5 of a component's range; two steps
# and a margin of 2.5.  A wrong sign or component in a flux is of order 1e-2.
TOL = 1e-4


def _state(n, ndim, axes, gamma):
    """A smooth random state around a fast flow, along `axes` (a permutation)."""
    rng = np.random.default_rng(5)
    x = [(np.arange(k) + 0.5) / k for k in n]
    Z, Y, X = np.meshgrid(x[2], x[1], x[0], indexing="ij")
    g = [X, Y, Z]
    pert = lambda a: a * sum(np.sin(2 * np.pi * (g[axes[d]] + rng.random())) for d in range(3) if n[axes[d]] > 1)
    v0, B0 = (0.88, 0.25, -0.2), (0.4, -0.6, 0.5)
    V = [1 + pert(0.1), None, None, None, 0.4 + pert(0.05), None, None, None, pert(0.02)]
    for d in range(3):
        V[1 + axes[d]] = v0[d] + pert(0.01)
        V[5 + axes[d]] = B0[d] + pert(0.1)
    U0 = np.zeros(O.shape(n, ndim))
    O.interior(U0, n, ndim)[:] = W.srmhd_cons(V, gamma)
    return U0


def _oracle(U0, n, ndim, dx, gamma):
    """Two steps of the oracle, whose boxes hold at least as many cells as
    ghosts: a thinner one is the period of a wider box."""
    k = [-(-4 // n[d]) if d < ndim else 1 for d in range(3)]
    m = [k[d] * n[d] for d in range(3)]
    U = np.zeros(O.shape(m, ndim))
    O.interior(U, m, ndim)[:] = np.tile(O.interior(U0, n, ndim), (1, k[2], k[1], k[0]))
    res = O.srmhd_run(U, m, ndim, dx + [1.0] * (3 - ndim), 2, 0.3, gamma=gamma)
    return O.interior(res[0], m, ndim)[:, :n[2], :n[1], :n[0]], res[-1][-1][1]


@pytest.mark.parametrize("tm", [0, 1], ids=["ideal", "taub-mathews"])
@pytest.mark.parametrize("n,ndim,axes", [((33, 6, 5), 3, (0, 1, 2)), ((5, 33, 6), 3, (1, 2, 0)),
                                         ((6, 5, 33), 3, (2, 0, 1)), ((1, 2, 17), 3, (2, 1, 0)),
                                         ((9, 40, 1), 2, (1, 0, 2)), ((40, 9, 1), 2, (0, 1, 2))])
def test_mixed_sweeps(n, ndim, axes, tm):
    gamma = 0.0 if tm else 4.0 / 3.0
    n = list(n)
    U0 = _state(n, ndim, axes, gamma)
    dx = [1 / max(n)] * ndim
    got, gd, st = gpu_run(U0, n, ndim, dx, 2, 0.3, precision=1, gamma=gamma, physics=1, eos=tm)
    assert st == 0
    ref, ch = _oracle(U0, n, ndim, dx, gamma)
    e = maxrel(O.interior(got, n, ndim), ref, ch)
    assert np.all(e <= TOL), e
