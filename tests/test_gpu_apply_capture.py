"""seed_apply inside a stream capture: graphs of D and D^H use no work space of the context,
and graphs of A keep theirs when the context grows."""
import numpy as np
import pytest

from paper_0810_0330_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# (16384 sites: the FP64 fixed-point form outside a capture; 65536: the FP32 form through tiled columns;
#  a partial last tile, and columns that are not 16-byte aligned)
@pytest.mark.parametrize("dims,op,pad,launches", [
    ((8, 16, 8, 16), 1, 0, 1), ((8, 16, 8, 16), 2, 0, 1), ((8, 16, 8, 16), 0, 0, None),
    ((16, 16, 16, 16), 4, 0, 1), ((16, 16, 16, 16), 5, 0, 1), ((16, 16, 16, 16), 4, 1, 1),
    ((17, 15, 17, 16), 5, 1, 1), ((16, 16, 16, 16), 3, 0, None)])
def test_captured_apply_outlives_growth(seedlib, dims, op, pad, launches):
    """FP32: the same bits as outside a capture; FP64: D (or D^H D) of each form is within
    2e-15 (4e-15) of the exact one (9 terms of up to 8 roundings, once or twice)."""
    low = op >= 3
    dt = torch.complex64 if low else torch.complex128
    n, cols = 12 * I.lattice_sites(dims), 3
    rng = np.random.default_rng(op)
    src = torch.complex(*torch.from_numpy(rng.standard_normal((2, cols, n))).cuda()).to(dt)
    U = torch.from_numpy(I.random_su3_links(dims, 0.3, seed=5)).cuda()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        ctx = seedlib.seed_create_wilson(dims, 0.155, U, seedlib.seed_params_default(m_max=2, precision=int(low)), bc_t=1)
        X = torch.zeros(cols, n + pad, dtype=dt, device="cuda")
        Y = torch.zeros_like(X)
        x, y = X[:, :n], Y[:, :n]
        seedlib.seed_apply(ctx, op, x.t(), y.t())   # room for `cols` columns
        s.synchronize()
        before = seedlib.seed_get_stats(ctx)["kernel_launches"]
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            seedlib.seed_apply(ctx, op, x.t(), y.t())
        if launches is not None:   # the operator alone: nothing that could use work space
            assert seedlib.seed_get_stats(ctx)["kernel_launches"] - before == launches
        wide = torch.zeros(2 * cols, n, dtype=dt, device="cuda")
        wide[cols:] = src
        out = torch.zeros_like(wide)
        seedlib.seed_apply(ctx, op, wide.t(), out.t())   # the context grows
        x.copy_(src)
        g.replay()
        s.synchronize()
        got, ref = y.clone(), out[cols:]
    if low:
        assert torch.equal(got, ref)
    else:
        assert torch.linalg.vector_norm(got - ref) <= (8e-15 if op == 0 else 4e-15) * torch.linalg.vector_norm(ref)
    seedlib.seed_destroy(ctx)
