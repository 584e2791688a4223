"""The Taub-Mathews gas's own mixed sweeps and segment rule: a patch stepped alone,
in short segments, and beside a large one, in long ones, gives the same bits."""
import numpy as np
import pytest

from tests.test_gpu_srmhd_sweeps import _state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ndim", [((9, 11, 7), 3), ((33, 34, 1), 2), ((1, 2, 19), 3)])
def test_segments_do_not_change_the_step(n, ndim):
    import torch
    from paper_1110_0740_gb300 import ctu
    big = (64, 64, 64) if ndim == 3 else (512, 256, 1)
    cfg = ctu.make_config(ndim=ndim, gamma=4 / 3, recon=ctu.CTU_LINEAR_MC, precision=ctu.CTU_MIXED, cfl=0.3,
                          physics=ctu.CTU_SRMHD, predictor=ctu.CTU_MUSCL_HANCOCK, riemann=ctu.CTU_HLL,
                          eos=ctu.CTU_EOS_TM)
    A = _state(list(n), ndim, (0, 1, 2), 0.0).reshape(9, -1)
    B = _state(list(big), ndim, (0, 1, 2), 0.0).reshape(9, -1)
    out = []
    for pool, boxes in ((A, [n]), (np.concatenate([A, B], axis=1), [n, big])):
        U = torch.from_numpy(np.ascontiguousarray(pool)).cuda()
        Uo = torch.zeros_like(U)
        P = ctu.make_patches([(b, [1 / 40] * 3, 0 if i == 0 else A.shape[1]) for i, b in enumerate(boxes)])
        ctx = ctu.Ctx(cfg)
        ctx.fill_periodic(U, U.shape[1], P)
        ctx.step(U, Uo, U.shape[1], P, torch.tensor([2e-3, 1.0], dtype=torch.float64, device="cuda"))
        assert ctx.status_sync() == 0
        out.append(Uo[:, :A.shape[1]].cpu().numpy())
    assert np.array_equal(*out)
