"""The float32 sweeps of the projected SVD with warps that have no blocks of M (K = J b up to about 56) and without: every
pass over the same matrix gives the same bits, in a cluster and in one CTA."""
import numpy as np
import pytest

from oracle import svt as osvt
from svt_inputs import planted_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block,steps", [(8, 2), (8, 3), (8, 5), (16, 3), (8, 7), (16, 4), (24, 3), (32, 4)])
@pytest.mark.parametrize("cluster", [0, 1])
def test_same_bits_every_time(cuda, block, steps, cluster):
    from paper_0810_3286_gb300 import Solver
    p = planted_problem(190, 160, 4, 5600, seed=3)
    tau = p.tau_default()
    y = 1.6 * tau / osvt.spectral_norm(p.n1, p.n2, p.rows, p.cols, p.vals) * p.vals

    def shrink():
        with Solver(p.n1, p.n2, p.rows, p.cols, p.vals, lanczos_tol=1e-9, block=block, lanczos_steps=steps,
                    jacobi_cluster=cluster) as s:
            s.set_Y(y)
            s.shrink(tau)
            return s.factors()

    first = shrink()
    assert first[1].size >= 1
    for _ in range(8):
        assert all(np.array_equal(a, b) for a, b in zip(first, shrink()))
