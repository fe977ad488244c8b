"""Stops of the one-launch reorthogonalizing seed run that only extreme values reach."""
import numpy as np
import pytest

from test_gpu_parity import csr_ctx, dev_cols

pytestmark = pytest.mark.gpu


def overflowing_matrix(d=8, m=6.0e307, t=0.25):
    """b = e_0: v_2 = (0, 1, ..., 1) / sqrt(d) after the first step, and A v_2 and alpha_2 are finite but
    f = A v_2 - alpha_2 v_2 - beta_1 v_1 overflows in its row 1."""
    A = np.full((d + 1, d + 1), 0.2 * m)
    A[0, 1:] = A[1:, 0] = t
    A[1, 1:] = A[1:, 1] = -m
    A[0, 0] = 1.0
    A[range(2, d + 1), range(2, d + 1)] = 2.0 * m
    return A


def test_overflow_case_is_what_it_says():
    A = overflowing_matrix()
    v1 = np.eye(9)[0]
    f = A @ v1 - v1
    beta = np.linalg.norm(f)
    v2 = f / beta
    u = (A @ f) / beta - beta * v1
    alpha = v2 @ u
    assert np.all(np.isfinite(u)) and np.isfinite(alpha) and alpha - beta * beta > 0
    with np.errstate(over="ignore"):
        assert np.isinf(u - alpha * v2)[1]


@pytest.mark.parametrize("nrhs", [1, 2])
@pytest.mark.parametrize("passes", [1, 2])
@pytest.mark.parametrize("kernel_path", [0, 1])
def test_non_finite_norm_is_not_convergence(seedlib, kernel_path, passes, nrhs):
    """A reorthogonalizing step whose ||f|| is not a number: SEED_ENOTSPD at the next step on
    every path, never a converged solve."""
    A = overflowing_matrix()
    n = A.shape[0]
    rp = np.arange(0, n * n + 1, n, dtype=np.int32)
    ci = np.tile(np.arange(n, dtype=np.int32), n)
    B = np.zeros((n, nrhs))
    B[0] = 1.0
    ctx = csr_ctx(seedlib, rp, ci, A.ravel().copy(), m_max=12, reorth_freq=1, reorth_passes=passes, tol_seed=1e-12,
                  kernel_path=kernel_path)
    with pytest.raises(seedlib.SeedError) as e:
        seedlib.seed_solve_first(ctx, dev_cols(B), dev_cols(np.zeros_like(B)))
    assert e.value.status == seedlib.SEED_ENOTSPD, e.value
    seedlib.seed_destroy(ctx)
