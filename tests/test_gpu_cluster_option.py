"""jacobi_cluster concerns the projected SVD of float64 contexts."""
import numpy as np
import pytest

from svt_inputs import config_problem

pytestmark = pytest.mark.gpu


def test_float32_contexts_take_the_cluster_whatever_the_option(cuda):
    """The same bits and so the same grouping of sums: one CTA in place of eight doubled the time of float32 solves of rank 30."""
    from paper_0810_3286_gb300 import Solver
    p = config_problem("plain_fp64_200", 0)
    out = []
    for option in (0, 1):
        with Solver(p.n1, p.n2, p.rows, p.cols, p.vals, precision="fp32", block=32, jacobi_cluster=option, k_max=8) as s:
            s.set_profile(["jacobi"])
            s.solve(p.tau_default(), p.delta_default(), 1e-4, 27, raise_on_nonconvergence=False)
            n, ms, _, _ = s.profile()["jacobi"]
            out.append((s.get_Y(), s.factors(), 1e3 * ms / n))
    print("us a projected SVD: %.0f, %.0f" % (out[0][2], out[1][2]))
    assert np.array_equal(out[0][0], out[1][0])
    assert all(np.array_equal(a, b) for a, b in zip(out[0][1], out[1][1]))
    assert out[1][2] <= 1.3 * out[0][2]
