"""Blocks of 8 columns on both sides of the line between float64 instructions and digit products (24 rows a CTA of two per SM),
with and without remainders, on capped grids too."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,grid", [(2425, 0), (2433, 0), (5003, 0), (7295, 0), (7296, 0), (7297, 0), (961, 40), (960, 40), (190, 8),
                                    (1500, 130)])
def test_blocks_of_8_columns(cuda, m, grid):
    """Orthonormality of the singular vectors to 1e-13 and X to 1e-8, as in the tests of the other sizes (the residual
    tolerance is 1e-11 sigma_1, the gaps are 0.1 sigma_1 and more)."""
    from paper_0810_3286_gb300 import Solver
    rng = np.random.default_rng(m)
    n = 48
    U, V = np.linalg.qr(rng.standard_normal((m, 3)))[0], np.linalg.qr(rng.standard_normal((n, 3)))[0]
    Y = (U * [1.0, 0.9, 0.8]) @ V.T + 1e-2 * rng.standard_normal((m, n)) / np.sqrt(m + n)
    u, d, vt = np.linalg.svd(Y, full_matrices=False)
    rows, cols = np.divmod(np.arange(m * n, dtype=np.int32), np.int32(n))
    with Solver(m, n, rows, cols, Y.ravel(), precision="fp64", block=8, ell=1, orth_grid=grid, lanczos_tol=1e-11) as s:
        s.configure(0.5, 1.0, 1e-4, 3, 1)
        s.set_Y(Y.ravel())
        s.shrink(0.5)
        Ug, dg, Vg = s.factors()
    assert len(dg) == 3
    for w in (Ug, Vg):
        assert np.abs(w.T @ w - np.eye(3)).max() <= 1e-13
    X = (u[:, :3] * (d[:3] - 0.5)) @ vt[:3]
    assert np.linalg.norm((Ug * dg) @ Vg.T - X) <= 1e-8 * np.linalg.norm(X)
