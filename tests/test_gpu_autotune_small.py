"""ctu_autotune leaves a step no slower than it found it, on small batches too,
where the default takes segments shorter than any it tries."""
import numpy as np
import pytest

import oracle as O
from paper_1110_0740_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _time(ctx, U, Uo, P, d):
    import torch
    best = []
    for _ in range(12):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        ctx.step(U, Uo, U.shape[1], P, d)
        ctx.step(U, Uo, U.shape[1], P, d)
        b.record()
        torch.cuda.synchronize()
        best.append(a.elapsed_time(b))
    return min(best)


# Pairs are kept only where their step beats the default's, each the best of six;
# two such timings of one configuration differ by less than 5%.
@pytest.mark.parametrize("n,ndim", [((128, 128, 1), 2), ((32, 32, 32), 3)], ids=["2d", "3d"])
def test_tuned_is_no_slower(n, ndim):
    import torch
    from paper_1110_0740_gb300 import ctu
    F = W.mhd_turb_2d(128, seed=1) if ndim == 2 else W.mhd_blast_3d(32, seed=1, kmax=3)
    U = torch.from_numpy(np.ascontiguousarray(F).reshape(9, -1)).cuda()
    assert U.shape[1] == np.prod(O.shape(list(n), ndim)[1:])
    Uo = torch.zeros_like(U)
    P = ctu.make_patches([(n, [1 / n[0]] * 3, 0)])
    ctx = ctu.Ctx(ctu.make_config(ndim=ndim, precision=ctu.CTU_FP64, cfl=0.3))
    d = torch.zeros(2, dtype=torch.float64, device="cuda")
    ctx.fill_periodic(U, U.shape[1], P)
    ctx.dt(U, U.shape[1], P, d)
    before = _time(ctx, U, Uo, P, d)
    ctx.autotune(U, Uo, U.shape[1], P, d)
    assert _time(ctx, U, Uo, P, d) <= 1.1 * before
