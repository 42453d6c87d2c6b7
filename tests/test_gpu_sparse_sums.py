"""Float32 sparse products of long segments: the chains of float32 additions stay short."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("b", [8, 16, 32, 48, 64])
@pytest.mark.parametrize("length", [700, 1000])
def test_float32_chains(cuda, b, length):
    """Equal entries of 1 + 31 2^-23, the bound in units of 2^-23 of the sum.  A float32 sum of 64 and more loses the 31 units of
    every further addition, all in one direction: 15 units for a chain of 125 additions, 27 for one of 500.  Chains of at most 24
    additions (16, times 3/2 where a length is no multiple of the piece) stay below 32, where an addition is off by at most 8
    units (4 below 16, 2 below 8, ...): 5 on average.  One addition that joins a lane's two sums and at most four between
    lanes, half a unit each, make it 7.5; asked are 9."""
    torch = cuda
    from paper_0810_3286_gb300 import Solver
    n1, n2 = 4200, 1100
    lens = np.full(n1, length)
    lens[::7] -= 13
    rows = np.repeat(np.arange(n1, dtype=np.int32), lens)
    cols = np.concatenate([np.arange(k, dtype=np.int32) for k in lens])
    c = 1.0 + 31 * 2.0 ** -23
    y = np.full(rows.size, c)
    with Solver(n1, n2, rows, cols, y, precision="fp32") as s:
        s.set_Y(y)
        W = torch.empty((n1, b), dtype=torch.float64, device="cuda")
        Z = torch.empty((n2, b), dtype=torch.float64, device="cuda")
        s.apply_Y(torch.ones((n2, b), dtype=torch.float64, device="cuda"), W)
        s.apply_Yt(torch.ones((n1, b), dtype=torch.float64, device="cuda"), Z)
        torch.cuda.synchronize()
    ref_w = (c * lens)[:, None]
    ref_z = (c * np.bincount(cols, minlength=n2))[:, None]
    assert np.abs(W.cpu().numpy() / ref_w - 1.0).max() <= 9 * 2.0 ** -23
    Z = Z.cpu().numpy()
    assert np.abs(Z - ref_z).max() <= 9 * 2.0 ** -23 * ref_z.max()
