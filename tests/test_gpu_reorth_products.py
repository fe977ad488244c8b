"""Precision of the one-launch reorthogonalizing seed run's products with the basis."""
import numpy as np
import pytest

from paper_0810_0330_gb300 import inputs as I
from test_gpu_parity import csr_ctx, dev_cols

pytestmark = pytest.mark.gpu

# FP64 sums in the run's shapes (16, 32, 64 rows per block), emulated on random unit vectors against
# exact sums: rms error of a product 2.9e-18 to 3.2e-18 at 2304 to 9216 rows.  The basis is
# orthogonal to what its products are: the rounding of its own entries adds 1e-18 at most.
FP64_SUMS = 3.2e-18


def off_diagonal_rms(seedlib, side, kernel_path, source, cols, passes=2):
    rp, ci, v = I.laplacian_2d_csr(*side)
    n = side[0] * side[1]
    B = I.gaussian_rhs(n, 1, seed=7)
    if source == "point":
        B[:] = 0.0
        B[n // 2 + side[0] // 3] = 1.0
    ctx = csr_ctx(seedlib, rp, ci, v, m_max=1000, reorth_freq=1, reorth_passes=passes, tol_seed=1e-12,
                  kernel_path=kernel_path, keep_basis=1)
    info = seedlib.seed_solve_first(ctx, dev_cols(B), dev_cols(np.zeros_like(B)))
    m = info[0]["iters"]
    V = np.ascontiguousarray(seedlib.seed_get_basis(ctx, m).T).astype(np.longdouble)
    seedlib.seed_destroy(ctx)
    late = V[-cols:]   # the last columns against all before them
    G = late @ V.T
    k = np.arange(m - cols, m)
    o = G[k[:, None] > np.arange(m)[None, :]].astype(float)
    return m, float(np.sqrt(np.mean(o * o)))


# 16, 32 and 64 rows per block, ragged last blocks; 96 x 96: late columns past those in shared memory
@pytest.mark.parametrize("side,source", [((48, 48), "gauss"), ((49, 47), "point"), ((64, 64), "gauss"),
                                         ((64, 64), "point"), ((71, 53), "gauss"), ((96, 96), "gauss")])
def test_products_no_less_precise_than_fp64_sums(seedlib, side, source):
    m, rms = off_diagonal_rms(seedlib, side, 0, source, 60)
    _, steps = off_diagonal_rms(seedlib, side, 1, source, 60)
    print("off-diagonal rms: one launch %.2e, step kernels (FP64) %.2e, %d steps" % (rms, steps, m))
    assert rms <= max(steps, FP64_SUMS), (rms, steps)
    if side == (96, 96):
        assert m > 200   # more columns than a block of 64 rows holds
