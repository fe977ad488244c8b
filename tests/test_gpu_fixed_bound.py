"""The stated accuracy of the fixed-point Wilson operator where components of a site differ
widely in size: a bound by site, with FP64 accuracy by component in the other forms."""
import numpy as np
import pytest

from paper_0810_0330_gb300 import inputs as I
from test_gpu_fixed import CLD, LD, dirac, dslash_bound, on_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def split_colours(vol, cols, split, seed):
    """Spinors whose colour 1 is `split` times its colours 0 and 2."""
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((cols, vol, 4, 3)) + 1j * rng.standard_normal((cols, vol, 4, 3))
    x[..., 1] *= split
    return x.reshape(cols, -1)


@pytest.mark.parametrize("split", [2.0 ** -70, 2.0 ** -30])
@pytest.mark.parametrize("dims,cols", [((4, 4, 4, 4), 1), ((4, 4, 4, 6), 20)])
def test_decoupled_colours(seedlib, dims, cols, split):
    """Unit links: colours decouple.  Fixed point: within the bound by site (derived in
    test_gpu_fixed), which says nothing about colour 1; seed_wilson_apply_noalloc, in FP64: every
    colour to its own scale.  The terms of D add up to (1 + 16 kappa) = 3 times the colour's largest value; 9
    terms of up to 8 roundings: 72 x 3 units of 2^-53 for D, 2 x 72 x 9 for D^H D, times sqrt 2 for a
    complex error."""
    vol, kappa = int(np.prod(dims)), 0.125
    U, x = I.unit_links(dims), split_colours(vol, cols, split, 3)
    y = on_gpu(seedlib, dims, kappa, 1, U, x, 0)
    X = torch.from_numpy(x).cuda().t()
    W = torch.empty_like(X.t()).t()
    seedlib.seed_wilson_apply_noalloc(dims, kappa, torch.from_numpy(U).cuda(), X, W, bc_t=1)
    w = W.t().cpu().numpy()
    for j in (0, cols - 1):
        t, tau = dslash_bound(dims, kappa, 1, U, x[j], 1)
        ref, tol = dslash_bound(dims, kappa, 1, U, t, -1)
        tol = tol + 17 * dirac(dims, kappa, 1, U, tau.astype(CLD).ravel(), 1)[1][:, None]
        assert np.all(np.abs(y[j] - ref).reshape(vol, 12) <= tol)
        e = np.abs(w[j] - ref).reshape(vol, 4, 3)
        for c in range(3):
            assert e[..., c].max() <= 1833 * LD(2) ** -53 * np.abs(x[j].reshape(vol, 4, 3)[..., c]).max(), (j, c)


def test_captured_d_is_in_fp64_on_a_large_lattice(seedlib):
    """From 16384 sites on D and D^H are in fixed point, but in FP64 arithmetic in a capture:
    colour 1 to its own scale (72 x 3 x sqrt 2 units, as above)."""
    dims, kappa, split = (8, 16, 8, 16), 0.125, 2.0 ** -70
    vol = int(np.prod(dims))
    U, x = I.unit_links(dims), split_colours(vol, 1, split, 4)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        ctx = seedlib.seed_create_wilson(dims, kappa, torch.from_numpy(U).cuda(), seedlib.seed_params_default(m_max=2))
        X = torch.from_numpy(x).cuda().t()
        Y, Z = torch.empty_like(X.t()).t(), torch.empty_like(X.t()).t()
        for op, sign in ((1, 1), (2, -1)):
            seedlib.seed_apply(ctx, op, X, Z)
            s.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                seedlib.seed_apply(ctx, op, X, Y)
            g.replay()
            s.synchronize()
            ref, tol = dslash_bound(dims, kappa, 0, U, x[0], sign)
            assert np.all(np.abs(Z.t().cpu().numpy()[0] - ref).reshape(vol, 12) <= tol)
            e = np.abs(Y.t().cpu().numpy()[0] - ref).reshape(vol, 4, 3)
            for c in range(3):
                top = np.abs(x[0].reshape(vol, 4, 3)[..., c]).max()
                assert e[..., c].max() <= 306 * LD(2) ** -53 * top, (op, c)
        seedlib.seed_destroy(ctx)
