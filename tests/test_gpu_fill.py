"""ctu_fill_periodic against numpy's wrap padding, bit for bit: every ghost
region, boxes of fewer cells than ghosts (several wraps), 1-D to 3-D."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ndim", [((1, 1, 1), 1), ((9, 1, 1), 1), ((3, 5, 1), 2), ((130, 33, 1), 2), ((1, 1, 1), 3),
                                    ((2, 3, 1), 3), ((4, 7, 5), 3), ((33, 16, 9), 3)])
def test_fill_is_wrap_padding(n, ndim):
    import torch
    from paper_1110_0740_gb300 import ctu
    rng = np.random.default_rng(4)
    inner = rng.normal(size=(2, 9, n[2], n[1], n[0]))  # two patches
    pad = [(0, 0)] + [(4, 4) if d < ndim else (0, 0) for d in (2, 1, 0)]
    blocks = [np.pad(u, pad, constant_values=np.nan) for u in inner]
    size = blocks[0][0].size
    U = torch.from_numpy(np.concatenate([b.reshape(9, -1) for b in blocks], axis=1)).cuda()
    ctx = ctu.Ctx(ctu.make_config(ndim=ndim))
    ctx.fill_periodic(U, U.shape[1], ctu.make_patches([(n, [0.1] * 3, 0), (n, [0.1] * 3, size)]))
    got = U.cpu().numpy()
    for i, u in enumerate(inner):
        want = np.pad(u, pad, mode="wrap")
        assert np.array_equal(got[:, i * size:(i + 1) * size].reshape(want.shape), want)
