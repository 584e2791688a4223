"""The launch shape of an untuned step (segment length from the whole batch,
row widths from the patch shape) changes nothing: a patch stepped alone, where
short segments fill the chip, and beside a large one, where they are long, gives
the same bits, and the float64 result is the oracle's within 1e-11 (relative L1
and elementwise).  Shapes at the edges of the tiles: one cell, a width of one
full row and one cell more, odd ones, 1-D to 3-D."""
import numpy as np
import pytest

import oracle as O
from paper_1110_0740_gb300 import workloads as W
from tests.gpu_util import l1rel, maxrel

pytestmark = pytest.mark.gpu

SHAPES = {1: [(1, 1, 1), (131, 1, 1)], 2: [(1, 3, 1), (33, 17, 1), (130, 67, 1)],
          3: [(1, 1, 1), (8, 8, 8), (16, 5, 7), (33, 34, 9), (65, 18, 31)]}
BIG = {1: (4096, 1, 1), 2: (1024, 1024, 1), 3: (128, 128, 128)}


def _state(n, ndim):
    src = O.interior(W.mhd_blast_3d(32, seed=3, kmax=3), [32] * 3, 3) if ndim == 3 else \
        O.interior(W.mhd_turb_2d(32, seed=3), [32, 32, 1], 2)
    sh = O.shape(list(n), ndim)
    ix = [(np.arange(s) - 4) % k if k > 1 else np.zeros(s, int) for s, k in zip(sh[1:], src.shape[1:])]
    return np.ascontiguousarray(src[:, ix[0]][:, :, ix[1]][:, :, :, ix[2]])


def _step(pool, shapes, bases, ndim, precision, dt, ch):
    import torch
    from paper_1110_0740_gb300 import ctu
    U = torch.from_numpy(pool).cuda()
    Uo = torch.zeros_like(U)
    ctx = ctu.Ctx(ctu.make_config(ndim=ndim, recon=ctu.CTU_PPM, precision=precision, cfl=0.3))
    d = torch.tensor([dt, ch], dtype=torch.float64, device="cuda")
    ctx.step(U, Uo, U.shape[1], ctu.make_patches([(n, [1 / 32] * 3, b) for n, b in zip(shapes, bases)]), d)
    assert ctx.status_sync() == 0
    return Uo.cpu().numpy()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("ndim", [1, 2, 3])
def test_launch_shape_does_not_change_the_step(ndim, precision):
    big = _state(BIG[ndim], ndim)
    dt, ch = 5e-4, 15.0
    for n in SHAPES[ndim]:
        A = _state(n, ndim)
        alone = _step(A.reshape(9, -1).copy(), [n], [0], ndim, precision, dt, ch)
        pool = np.concatenate([A.reshape(9, -1), big.reshape(9, -1)], axis=1)
        both = _step(pool, [n, BIG[ndim]], [0, A[0].size], ndim, precision, dt, ch)
        assert np.array_equal(alone, both[:, :A[0].size]), n
        if precision == 0:
            ref, bad = O.mhd_step(A, list(n), ndim, [1 / 32] * 3, dt, ch, recon=1)
            assert bad == 0
            G, R = O.interior(alone.reshape(A.shape), list(n), ndim), O.interior(ref, list(n), ndim)
            assert l1rel(G, R, ch).max() < 1e-11 and maxrel(G, R, ch).max() < 1e-11, n
