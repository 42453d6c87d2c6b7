"""Projected matrices with infinities and NaNs among finite entries: an iterate whose Gram matrices overflow is reported
as SVT_ERR_NUMERIC for every size of the projected matrix, and the context solves again afterwards."""
import numpy as np
import pytest

from oracle import svt as osvt
from svt_inputs import planted_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block,steps", [(8, 2), (16, 3), (24, 3), (32, 4)])
@pytest.mark.parametrize("cluster", [0, 1])
@pytest.mark.parametrize("kind", ["all", "one"])
def test_overflowing_iterate(cuda, block, steps, cluster, kind):
    from paper_0810_3286_gb300 import Solver, SVTError
    p = planted_problem(190, 160, 4, 5600, seed=3)
    tau = p.tau_default()
    y = 1.6 * tau / osvt.spectral_norm(p.n1, p.n2, p.rows, p.cols, p.vals) * p.vals
    bad = y * 1e200 if kind == "all" else np.where(np.arange(y.size) == 77, 1e200, y)
    with Solver(p.n1, p.n2, p.rows, p.cols, p.vals, block=block, lanczos_steps=steps, jacobi_cluster=cluster) as s:
        s.configure(tau)
        for _ in range(2):
            s.set_Y(bad)
            with pytest.raises(SVTError) as ei:
                s.shrink(tau)
            assert ei.value.status == 7   # SVT_ERR_NUMERIC
            s.configure(tau)
            s.set_Y(y)
            assert s.shrink(tau)[0] >= 1
