"""Orthonormality of the singular vectors of a tight shrink: the float64 accuracy of the bases' Gram and projection products,
which run as digit products on the tensor cores."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n", [(257, 130), (2100, 900)])
@pytest.mark.parametrize("block", [8, 16, 24, 32])
@pytest.mark.parametrize("kind", ["flat", "rows"])
def test_singular_vectors_are_orthonormal(cuda, m, n, block, kind):
    """The bases are orthonormal to a few 1e-15 (the last Gram's rounding, b 2^-53), the projected vectors to K 2^-53, and their
    product adds up to K 2^-53 a column: 1e-13 is several times their sum for K <= 128.  A product that is short of one of
    eight 8-bit digits in a column leaves 2^-48 of its scale, one short of two 2^-40 = 1e-12."""
    from paper_0810_3286_gb300 import Solver
    rng = np.random.default_rng(m + block)
    L = rng.standard_normal((m, 6))
    if kind == "rows":
        L *= 10.0 ** rng.uniform(-4, 0, (m, 1))
    U, V = np.linalg.qr(L)[0], np.linalg.qr(rng.standard_normal((n, 6)))[0]
    Y = (U * np.linspace(1.0, 0.7, 6)) @ V.T + 1e-2 * rng.standard_normal((m, n)) / np.sqrt(m + n)
    rows, cols = np.divmod(np.arange(m * n, dtype=np.int32), np.int32(n))
    with Solver(m, n, rows, cols, Y.ravel(), precision="fp64", block=block, lanczos_tol=1e-11) as s:
        tau = 0.35
        s.configure(tau, 1.0, 1e-4, 27, 1)
        s.set_Y(Y.ravel())
        s.shrink(tau)
        Ug, dg, Vg = s.factors()
    assert len(dg) == 6
    for w in (Ug, Vg):
        defect = np.abs(w.T @ w - np.eye(6)).max()
        print("%s b %d: %.1e" % (kind, block, defect))
        assert defect <= 1e-13
