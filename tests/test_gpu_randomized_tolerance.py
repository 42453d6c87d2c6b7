"""The randomized shrink engine's projected SVD in float32 contexts: to the accuracy of a Lanczos cycle there (1e-9), not to
float64 rounding."""
import pytest

from svt_inputs import config_problem

pytestmark = pytest.mark.gpu


def test_float32_takes_a_refinement_step_less(cuda):
    """Each refinement step squares the error: from float32 sweeps (1e-6), one step gives 1e-9 and two give 1e-15."""
    from paper_0810_3286_gb300 import Solver
    p = config_problem("plain_fp64_200", 0)
    steps = {}
    for precision in ("fp64", "fp32"):
        with Solver(p.n1, p.n2, p.rows, p.cols, p.vals, precision=precision, shrink_engine="randomized", k_max=40) as s:
            s.solve(p.tau_default(), p.delta_default(), 1e-4, 20, raise_on_nonconvergence=False)
            c = s.counters()
        steps[precision] = c["jacobi_sweeps"] / c["svd_calls"]
    print("sweeps and steps a projected SVD: float64 %.2f, float32 %.2f" % (steps["fp64"], steps["fp32"]))
    assert steps["fp32"] <= steps["fp64"] - 0.5
