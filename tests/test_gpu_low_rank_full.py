"""Solves of fully observed low-rank matrices: the projected matrices have null singular values (float64) or values at the
rounding of the products (float32), so that the leading block spans many orders of magnitude.  With P_Omega the identity
every iterate is U diag(y - tau)_+ V^T with y <- y + delta (sigma - (y - tau)_+) on the singular values sigma of M
(Algorithm 1, eq. (2.2)); k0 steps of it give the kick."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _closed_form(sigma, m, n, k_max, eps=1e-4):
    tau, delta = 5.0 * np.sqrt(m * n), 1.2
    y = np.ceil(tau / (delta * sigma[0])) * delta * sigma
    for k in range(1, k_max + 1):
        x = np.maximum(y - tau, 0.0)
        if np.linalg.norm(sigma - x) <= eps * np.linalg.norm(sigma):
            break
        y = y + delta * (sigma - x)
    return k, x


@pytest.mark.parametrize("m,n,r", [(300, 300, 5), (260, 180, 12), (400, 390, 30)])
@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("noise", [0.0, 1e-5])
def test_full_low_rank(cuda, m, n, r, precision, noise):
    """On every one of several solves (each starts from other random columns).  float64: the closed form's iterations, and X
    to the Lanczos tolerance of 1e-6 sigma_1, with a factor 2.  float32 and bfloat16: X is M to the stop's 1e-4, with a
    factor 2 for the rounding of the products."""
    from paper_0810_3286_gb300 import Solver
    rng = np.random.default_rng(m + r)
    M = rng.standard_normal((m, r)) @ rng.standard_normal((r, n)) + noise * rng.standard_normal((m, n))
    u, sigma, vt = np.linalg.svd(M, full_matrices=False)
    k, x = _closed_form(sigma, m, n, 60)
    rows, cols = (a.ravel().astype(np.int32) for a in np.indices((m, n)))
    X = (u * x) @ vt
    with Solver(m, n, rows, cols, M.ravel(), precision=precision, k_max=60, max_cycles=200) as s:
        for _ in range(5):
            res = s.solve(0.0, 0.0, 1e-4, 64)
            U, d, V = s.factors()
            if precision == "fp64":
                assert res["iterations"] == k and res["rank"] == (x > 0).sum()
                assert np.linalg.norm((U * d) @ V.T - X) <= 2e-6 * np.linalg.norm(X)
            else:
                assert np.linalg.norm((U * d) @ V.T - M) <= 2e-4 * np.linalg.norm(M)
