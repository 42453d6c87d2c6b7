"""Workspaces of a context: the scratch of the orthonormalisation and of the projected SVD is one buffer, and one set of partial
Grams on large grids."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,limit", [(100, 120, 1.3e6), (3000, 2500, 13e6)])
def test_workspace_bytes(cuda, m, n, limit):
    """The bases take 8 (m + n) 160 bytes, two Ritz blocks 8 (m + n) 128, the factors 8 (2 m + n) 65 and a few matrices of
    128 x 128 and 160 x 32 0.6 MB; the entries of Omega next to nothing.  What is left is the scratch: 304 partial Grams of 160 x
    32 float64 (12.5 MB), 1.2 MB on small problems.  Before, 24.9 MB and another 1.1 MB, in construction time too."""
    torch = cuda
    from paper_0810_3286_gb300 import Solver
    sizes = []

    def alloc(nbytes):
        sizes.append(int(nbytes))
        return torch.cuda.caching_allocator_alloc(int(nbytes))

    rng = np.random.default_rng(0)
    ids = np.sort(rng.choice(m * n, 2 * (m + n), replace=False))
    Solver(m, n, (ids // n).astype(np.int32), (ids % n).astype(np.int32), rng.standard_normal(ids.size), precision="fp64",
           allocator=(alloc, torch.cuda.caching_allocator_delete)).close()
    rest = sum(sizes) - 8 * (m + n) * 288 - 8 * (2 * m + n) * 65 - 64 * ids.size
    print("%d allocations, %.2f MB, scratch and small %.2f MB" % (len(sizes), sum(sizes) / 1e6, rest / 1e6))
    assert rest <= limit + 1.0e6
