"""Small reorthogonalizing problems side by side in a batch: two blocks of different
problems share an SM there, and every problem gets the bits of its solo solve."""
import numpy as np
import pytest

from paper_0810_0330_gb300 import inputs as I
from test_gpu_parity import csr_ctx

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sides", [(64, 64, 64), (96, 96), (48, 64, 96, 30)])
def test_batch_of_reorthogonalizing_runs_equals_solo(seedlib, sides):
    kw = dict(m_max=1000, reorth_freq=1, tol_seed=1e-12, tol_rest=1e-8)
    ctxs, Bs, Xs = [], [], []
    for q, side in enumerate(sides):
        rp, ci, v = I.laplacian_2d_csr(side, side)
        ctxs.append(csr_ctx(seedlib, rp, ci, v, **kw))
        Bs.append(torch.from_numpy(np.ascontiguousarray(I.gaussian_rhs(side * side, 3, seed=q).T)).cuda().t())
        Xs.append(torch.zeros_like(Bs[-1].t()).t())
    seedlib.seed_batch_solve(ctxs, Bs, Xs)
    torch.cuda.synchronize()
    for ctx, B, X in zip(ctxs, Bs, Xs):
        Y = torch.zeros_like(B.t()).t()
        seedlib.seed_solve_first(ctx, B, Y)
        seedlib.seed_solve_rest(ctx, B, Y)
        torch.cuda.synchronize()
        assert torch.equal(X, Y)
        seedlib.seed_destroy(ctx)
