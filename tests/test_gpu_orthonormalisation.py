"""The cooperative block orthonormalisation inside a shrink, against the dense SVD.

The residual tolerance is 1e-10 sigma_1 and the wanted singular values are 0.05 sigma_1 apart from each other and from
tau, so X = D_tau(Y) is good to about 1e-10 sqrt(r) / 0.05 < 1e-8 of its norm.
"""
import numpy as np
import pytest

from svt_inputs import config_problem
from oracle.sparse import sample_X

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,grid", [(49, 48, 0), (65, 63, 0), (127, 130, 0), (257, 96, 1), (400, 130, 3), (521, 300, 4)])
@pytest.mark.parametrize("block", [8, 16, 24, 32])
@pytest.mark.parametrize("kind", ["flat", "rows", "large", "small"])
def test_shrink_by_chunk_height_and_block(cuda, m, n, grid, block, kind):
    """Chunks of 8 and 16 rows with and without remainders, chunks of over 64 (orth_grid), every block size; rows that
    differ by 10^4 in size; entries near 10^+-60."""
    from paper_0810_3286_gb300 import Solver
    rng = np.random.default_rng(m + n + block)
    L = rng.standard_normal((m, 3))
    if kind == "rows":
        L *= 10.0 ** rng.uniform(-4, 0, (m, 1))
    U, V = np.linalg.qr(L)[0], np.linalg.qr(rng.standard_normal((n, 3)))[0]
    Y = (U * [1.0, 0.9, 0.8]) @ V.T + 1e-3 * rng.standard_normal((m, n)) / np.sqrt(m + n)
    Y *= {"large": 1e60, "small": 1e-60}.get(kind, 1.0)
    u, d, vt = np.linalg.svd(Y, full_matrices=False)
    tau = 0.5 * d[0]
    X = (u[:, :3] * (d[:3] - tau)) @ vt[:3]
    rows, cols = np.divmod(np.arange(m * n, dtype=np.int32), np.int32(n))
    with Solver(m, n, rows, cols, Y.ravel(), precision="fp64", block=block, orth_grid=grid, lanczos_tol=1e-10) as s:
        s.configure(tau, 1.0, 1e-4, 27, 1)
        s.set_Y(Y.ravel())
        s.shrink(tau)
        Ug, dg, Vg = s.factors()
    assert len(dg) == 3
    assert np.linalg.norm((Ug * dg) @ Vg.T / d[0] - X / d[0]) <= 1e-8 * np.linalg.norm(X / d[0])


@pytest.mark.parametrize("seed", [0, 1])
def test_dependent_blocks_keep_the_lanczos_relation(cuda, seed):
    """The rank policy's restarts from converged Ritz vectors make blocks with nearly dependent columns.  The default
    tolerance of 1e-6 sigma_1 bounds the error of X on Omega by about 1e-6, whatever the order of the sums."""
    from paper_0810_3286_gb300 import Solver
    p = config_problem("companion_2000", seed)

    def x(**kw):
        with Solver(p.n1, p.n2, p.rows, p.cols, p.vals, precision="fp64", **kw) as s:
            s.configure(p.tau_default(), p.delta_default(), 1e-4, 27, 5)
            s.step()
            U, d, V = s.factors()
        return sample_X(p.rows, p.cols, U * d, V)

    ref = x(lanczos_tol=1e-13)
    for kw in ({}, {"orth_grid": 8}, {"orth_grid": 40}, {"orth_grid": 77}, {"fused_orth": False}, {"orth_repass": -1.0}):
        assert np.linalg.norm(x(**kw) - ref) <= 1e-6 * np.linalg.norm(ref), kw
