"""The one-launch reorthogonalizing seed run on the launch shapes its sister
file does not reach: 16 rows per block (a last block of one row, sixteen and one
right-hand sides, a matrix with rows too long for the row cache), and one block.
Checks and tolerances as there."""
import numpy as np
import pytest

from paper_0810_0330_gb300 import inputs as I
from test_gpu_parity import REL_X, compare_full, csr_ctx, dev_cols, host_cols, run_gpu, self_sensitivity

pytestmark = pytest.mark.gpu


def band_csr(n, half):
    """Diagonally dominant band matrix, 2 half + 1 entries per row."""
    i, j = np.meshgrid(np.arange(n), np.arange(-half, half + 1), indexing="ij")
    c = i + j
    ok = (c >= 0) & (c < n)
    v = np.where(j == 0, 2.0 * half + 0.05, -1.0)
    rp = np.concatenate([[0], np.cumsum(ok.sum(1))])
    return rp.astype(np.int32), c[ok].astype(np.int32), np.ascontiguousarray(v[ok])


@pytest.mark.parametrize("matrix,freq,passes,nrhs", [
    (I.laplacian_2d_csr(49, 49), 1, 2, 16),   # n = 2401: 151 blocks, the last with one row
    (I.laplacian_2d_csr(49, 49), 5, 1, 3),
    (band_csr(1000, 6), 1, 2, 2),             # 13 entries per row
    (I.laplacian_2d_csr(3, 4), 2, 2, 2),      # one block
])
def test_reorth_run_shapes(seedlib, orc, matrix, freq, passes, nrhs):
    rp, ci, v = matrix
    n = rp.shape[0] - 1
    B = I.gaussian_rhs(n, nrhs, seed=n)
    kw = dict(m_max=1000, reorth_freq=freq, reorth_passes=passes)
    ctx = csr_ctx(seedlib, rp, ci, v, tol_seed=1e-12, tol_rest=1e-8, keep_basis=1, **kw)
    info1, info2, Xs, X = run_gpu(seedlib, ctx, B)
    op = orc.Operator.csr(rp, ci, v)
    ref = orc.seed_solve_all(op, B, tol_seed=1e-12, tol_rest=1e-8, **kw)
    s_seed, s_final = self_sensitivity(orc, op, B, ref, cols=(1,), tol=1e-12, **kw)
    compare_full(ref, info1, info2, Xs.real, X.real, "n%d-f%d" % (n, freq),
                 seeded_tol=max(REL_X, 10 * s_seed), final_tol=max(REL_X, 10 * s_final))
    m = info1[0]["iters"]
    V = seedlib.seed_get_basis(ctx, m)
    assert np.abs(V.T @ V - np.eye(m)).max() < 1e-12
    seedlib.seed_destroy(ctx)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [127, 512, 513, 2049, 40001])
def test_lockstep_cg_kernels_ragged(seedlib, n, precision):
    """Lockstep CG as step kernels (several elements ahead per thread): lengths at the edges of
    a thread's four elements and a block's 512.  The claim checked is CG's own: every true
    residual, recomputed here in FP64 (its rounding is below 1e-14), meets the tolerance."""
    import scipy.sparse as sp
    rp, ci, v = band_csr(n, 3)
    A = sp.csr_matrix((v, ci, rp), shape=(n, n))
    B = I.gaussian_rhs(n, 3, seed=n)
    ctx = csr_ctx(seedlib, rp, ci, v, tol_seed=1e-10, tol_rest=1e-10, m_max=50, kernel_path=1, precision=precision)
    X = dev_cols(np.zeros_like(B))
    info = seedlib.seed_solve_cg(ctx, dev_cols(B), X)
    r = np.linalg.norm(B - A @ host_cols(X).real, axis=0) / np.linalg.norm(B, axis=0)
    assert all(i["converged"] for i in info) and np.all(r <= 1.01e-10), r
    seedlib.seed_destroy(ctx)
