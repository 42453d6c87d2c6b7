"""Sparse products whose segments differ much in length: shared by a CTA at every number of warps a segment, and not the time
of the whole product."""
import numpy as np
import pytest

from oracle import sparse as osp
from svt_inputs import random_dense

pytestmark = pytest.mark.gpu

# as in the tests of the segment lengths: chains of at most 24 + 8 additions, norm-wise
TOL = {"fp64": 1e-13, "fp32": 1.5e-6}


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n1,mean,b", [(600, 120, 16), (1900, 500, 48), (2500, 100, 16), (5000, 300, 32), (9000, 20, 6)])
def test_long_segments(cuda, precision, n1, mean, b):
    """Eight, four, two and one warps a segment; long neighbours at the start, in the middle and at the end (the last one short
    of a tile), lengths around the threshold of three mean segments a warp."""
    torch = cuda
    from paper_0810_3286_gb300 import Solver
    n2 = 9000
    rng = np.random.default_rng(n1)
    lens = rng.integers(0, 2 * mean, n1)
    lens[:3] = [9000, 0, 2500]
    mid = n1 // 2
    lens[mid:mid + 12] = [3 * mean * w + d for w in (1, 2, 4, 8) for d in (-1, 0, 1)]
    lens[-3:] = [4000, 5000, 1]
    lens = np.minimum(lens, n2)
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
        torch.cuda.synchronize()
    W, Z = W.cpu().numpy(), Z.cpu().numpy()
    for got, ref in ((W, osp.apply_Y(n1, rows, cols, y, V)), (Z, osp.apply_Yt(n2, rows, cols, y, U))):
        assert np.linalg.norm(got - ref) <= TOL[precision] * np.linalg.norm(ref)


def test_long_neighbours_do_not_stall(cuda):
    """10000 segments of 120, the last eight of 1000: a warp takes 44 us and more for each of those, the product without them
    46 us.  Shared by eight warps in eight CTAs they add about 10 us; asked is less than 0.8 of the product."""
    torch = cuda
    from paper_0810_3286_gb300 import Solver
    n1, n2, b = 10000, 20000, 16
    rng = np.random.default_rng(1)
    V = torch.from_numpy(random_dense((n2, b), 1)).cuda()
    W = torch.empty((n1, b), dtype=torch.float64, device="cuda")

    def us(lens):
        rows = np.repeat(np.arange(n1, dtype=np.int32), lens)
        cols = np.concatenate([np.sort(rng.choice(n2, k, replace=False)) for k in lens]).astype(np.int32)
        with Solver(n1, n2, rows, cols, rng.standard_normal(rows.size), precision="fp64") as s:
            best = 1e9
            for _ in range(8):
                a, z = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                for _ in range(20):
                    s.apply_Y(V, W)
                z.record()
                torch.cuda.synchronize()
                best = min(best, a.elapsed_time(z) / 20 * 1e3)
        return best

    lens = np.full(n1, 120)
    plain = us(lens)
    lens[-8:] = 1000
    skewed = us(lens)
    print("%.1f us, with eight long segments %.1f us" % (plain, skewed))
    assert skewed <= 1.8 * plain
