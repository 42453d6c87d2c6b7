"""The float64 fused update with and without staging copies: apart, in place, into an overlapping array; factors off a
16-byte boundary."""
import numpy as np
import pytest

from svt_inputs import random_dense, random_sparse_pattern

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [1, 2, 5, 10, 33, 64])
@pytest.mark.parametrize("out", ["apart", "in_place", "shifted"])
@pytest.mark.parametrize("off", [0, 1])
def test_sddmm_outputs(cuda, r, out, off):
    torch = cuda
    from paper_0810_3286_gb300 import Solver
    m, n = 611, 301
    rows, cols, vals = random_sparse_pattern(m, n, 25000, 4, empty_rows=(3,), dense_rows=(9,))
    nnz, delta = rows.size, 3.7
    y, Ut, V = random_dense(nnz, 5), random_dense((m, r), 6), random_dense((n, r), 7)
    e = vals - (Ut[rows] * V[cols]).sum(1)
    buf = torch.zeros(2 * nnz + 8, device="cuda", dtype=torch.float64)
    y_in = buf[:nnz]
    y_in.copy_(torch.from_numpy(y))
    y_out = {"apart": buf[nnz:2 * nnz], "in_place": y_in, "shifted": buf[3:nnz + 3]}[out]
    vb = torch.zeros(n * r + 1, device="cuda", dtype=torch.float64)
    Vd = vb[off:off + n * r].view(n, r)
    Vd.copy_(torch.from_numpy(V))
    with Solver(m, n, rows, cols, vals, precision="fp64") as s:
        res2 = s.sddmm_update(torch.from_numpy(Ut).cuda(), Vd, delta, y_in, y_out)
    ref = y + delta * e
    # sums of up to 64 products and a handful of operations, 2^-53 each
    assert np.linalg.norm(y_out.cpu().numpy() - ref) <= 1e-13 * np.linalg.norm(ref)
    assert abs(res2 - e @ e) <= 1e-12 * (e @ e)
