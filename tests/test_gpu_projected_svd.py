"""The projected SVD (float32 sweeps on T^T T, float64 refinement, one-sided finish) through svt_shrink, over the sizes
of the projected matrix: K = J b from one block of 8 to the capacity of 128, in a cluster and in one CTA, on the
spectra that take each of its paths.

Bounds: the singular values above tau to 1e-9 sigma_1 and X to 1e-8 (the Ritz tolerance 1e-9 sigma_1 over relative gaps of
a few per cent, as in test_shrink_matches_definition), float32 values to 1e-4 / 1e-3."""
import numpy as np
import pytest

from oracle import svt as osvt
from oracle.sparse import sample_X
from svt_inputs import planted_problem

pytestmark = pytest.mark.gpu


def _check(s, m, n, rows, cols, y, tau, sig_tol, x_tol):
    s.set_Y(y)
    r, sig = s.shrink(tau)
    U0, d0, V0, s_all = osvt.shrink(osvt.dense_from_omega(m, n, rows, cols, y), tau)
    assert r == d0.size and r >= 1
    assert np.abs(sig - (d0 + tau)).max() <= sig_tol * s_all[0]
    U, d, V = s.factors()
    assert np.abs(U.T @ U - np.eye(r)).max() <= 1e-6 and np.abs(V.T @ V - np.eye(r)).max() <= 1e-6
    x, x0 = sample_X(rows, cols, U * d, V), sample_X(rows, cols, U0 * d0, V0)
    assert np.linalg.norm(x - x0) <= x_tol * np.linalg.norm(x0)


@pytest.mark.parametrize("block,steps", [(8, 2), (8, 3), (8, 9), (16, 3), (16, 4), (24, 3), (24, 5), (32, 3), (32, 4)])
@pytest.mark.parametrize("cluster", [0, 1])
def test_projected_sizes(cuda, block, steps, cluster):
    from paper_0810_3286_gb300 import Solver
    p = planted_problem(190, 160, 4, 5600, seed=3)
    tau = p.tau_default()
    y = 1.6 * tau / osvt.spectral_norm(p.n1, p.n2, p.rows, p.cols, p.vals) * p.vals
    with Solver(p.n1, p.n2, p.rows, p.cols, p.vals, lanczos_tol=1e-9, block=block, lanczos_steps=steps,
                jacobi_cluster=cluster) as s:
        _check(s, p.n1, p.n2, p.rows, p.cols, y, tau, 1e-9, 1e-8)
    with Solver(p.n1, p.n2, p.rows, p.cols, p.vals, precision="fp32", block=block, lanczos_steps=steps,
                jacobi_cluster=cluster) as s:
        _check(s, p.n1, p.n2, p.rows, p.cols, y, tau, 1e-4, 1e-3)


@pytest.mark.parametrize("kind,scale", [("graded", 1.0), ("low_rank", 1.0), ("pairs", 1.0), ("pairs", 1e40),
                                        ("pairs", 1e-40)])
def test_spectra(cuda, kind, scale):
    """Full Omega: values that span more than a factor 100 in the leading block (the one-sided finish), an exactly
    low-rank iterate (null columns of T), and near-equal pairs, at ordinary and extreme scales."""
    from paper_0810_3286_gb300 import Solver
    m, n = 70, 64
    rng = np.random.default_rng(5)
    U, _ = np.linalg.qr(rng.standard_normal((m, n)))
    V, _ = np.linalg.qr(rng.standard_normal((n, n)))
    sv = {"graded": 10.0 ** (-0.4 * np.arange(n)), "low_rank": np.where(np.arange(n) < 5, 5.0 - np.arange(n), 0.0),
          "pairs": np.repeat(1.0 / (1.0 + 0.3 * np.arange(n // 2)), 2) * (1 + 1e-9 * np.arange(n))}[kind]
    Y = (U * sv) @ V.T * (100.0 * scale)
    rows, cols = (a.ravel().astype(np.int32) for a in np.indices((m, n)))
    tau = 100.0 * scale * {"graded": 0.03, "low_rank": 0.5, "pairs": 0.6}[kind]
    with Solver(m, n, rows, cols, Y.ravel(), lanczos_tol=1e-9) as s:
        _check(s, m, n, rows, cols, Y.ravel(), tau, 1e-9, 1e-8)
