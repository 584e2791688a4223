"""The tiled tagging kernel at each number of planes a block marches (it follows
from the batch's size) and on values at the edges of float32's range (zeros of
both signs, denormals, huge values, infinities, NaNs with every bit set): tags
and counts equal the oracle's."""
import numpy as np
import pytest

import oracle as O
from paper_1110_0740_gb300 import workloads as W
from tests.test_gpu_tag import EPS, _gpu_tag, _pool

pytestmark = pytest.mark.gpu
N = [35, 20, 37]  # ragged in x, y and z for 4, 8 and 16 planes
EDGE = [0.0, -0.0, 1e-320, 1e-40, -1e-38, 1e30, 3.4028235e38, -3.5e38, 1e130, 1e-200, 1e308, np.inf, -np.inf, np.nan]


def _block(seed):
    rng = np.random.default_rng(seed)
    U = W.mhd_blast_3d(48, seed=seed)[:, :N[2] + 8, :N[1] + 8, :N[0] + 8].copy()
    U[5] *= rng.random(U[5].shape) < 0.7  # zero field components are common
    flat = U[[0, 4, 5, 6, 7]]
    at = rng.integers(0, U[0].size, size=(5, 60))
    for q in range(5):
        v = rng.choice(EDGE, size=60)
        v[:3] = np.array([0x7FFFFFFFFFFFFFFF, 0xFFFFFFFFFFFFFFFF, 0xFFF8000000000000], dtype=np.uint64).view(np.float64)
        flat[q].reshape(-1)[at[q]] = v
    U[[0, 4, 5, 6, 7]] = flat
    return U


@pytest.mark.parametrize("copies", [1, 11, 17], ids=["4 planes", "8 planes", "16 planes"])
@pytest.mark.parametrize("kind", [0, 1, 2, 3])
def test_planes_and_edges(kind, copies):
    b = _block(3)
    with np.errstate(all="ignore"):
        t_ref, chi, _ = O.tag(b, N, 3, kind, EPS, 0.1)
        chi_r = float(np.nanmedian(O.interior(chi[None], N, 3)))
        t_ref, _, c_ref = O.tag(b, N, 3, kind, EPS, chi_r)
    pool, bases = _pool([b] * copies)
    tags, cnt, _ = _gpu_tag(pool, [(N, [0.1] * 3, base) for base in bases], 3, kind, EPS, chi_r, False)
    want = O.interior(t_ref[None], N, 3)
    for i, base in enumerate(bases):
        T = tags[base:base + b[0].size].reshape(b.shape[1:])
        assert np.array_equal(O.interior(T[None], N, 3), want)
        assert cnt[i] == c_ref
