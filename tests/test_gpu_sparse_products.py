"""Sparse products with one warp a segment: segments around the length from which a CTA shares them, ragged tails, every
column-group width, infinities."""
import numpy as np
import pytest

from oracle import sparse as osp
from svt_inputs import random_dense

pytestmark = pytest.mark.gpu

# float64: chains of up to 4200 / 64 + 8 additions, 2^-53 each, against sums of random signs (norm-wise 1e-13 is 10x that);
# float32: chains of up to 64 + 8, 2^-24 each, norm-wise sqrt(72) 2^-24 = 5e-7, and 3x
TOL = {"fp64": 1e-13, "fp32": 1.5e-6}


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("b", [2, 6, 8, 16, 24, 32, 64])
@pytest.mark.parametrize("n1", [8, 4500])
def test_segment_lengths(cuda, precision, b, n1):
    torch = cuda
    from paper_0810_3286_gb300 import Solver
    n2 = 4200
    rng = np.random.default_rng(b)
    lens = rng.integers(0, 40, n1)
    lens[:8] = [1023, 1024, 1025, 4200, 0, 1, 3, 2049]
    lens[-1] = max(lens[-1], 1)
    rows = np.repeat(np.arange(n1, dtype=np.int32), lens)
    cols = np.concatenate([np.sort(rng.choice(n2, k, replace=False)) for k in lens]).astype(np.int32)
    y = rng.standard_normal(rows.size)
    V, U = random_dense((n2, b), 1), random_dense((n1, b), 2)
    with Solver(n1, n2, rows, cols, y, precision=precision) as s:
        s.set_Y(y)
        W = torch.empty((n1, b), dtype=torch.float64, device="cuda")
        Z = torch.empty((n2, b), dtype=torch.float64, device="cuda")
        s.apply_Y(torch.from_numpy(V).cuda(), W)
        s.apply_Yt(torch.from_numpy(U).cuda(), Z)
        V[cols[0], 0] = np.inf
        W2 = torch.empty_like(W)
        s.apply_Y(torch.from_numpy(V).cuda(), W2)
        torch.cuda.synchronize()
        W2 = W2.cpu().numpy()
    V[cols[0], 0] = random_dense((n2, b), 1)[cols[0], 0]
    W, Z = W.cpu().numpy(), Z.cpu().numpy()
    for got, ref in ((W, osp.apply_Y(n1, rows, cols, y, V)), (Z, osp.apply_Yt(n2, rows, cols, y, U))):
        assert np.linalg.norm(got - ref) <= TOL[precision] * np.linalg.norm(ref)
    assert np.all(W[4] == 0.0)
    hit = np.zeros(n1, bool)
    hit[rows[cols == cols[0]]] = True
    assert np.all(np.isinf(W2[hit, 0])) and np.all(np.isfinite(W2[~hit])) and np.array_equal(W2[:, 1:], W[:, 1:])
