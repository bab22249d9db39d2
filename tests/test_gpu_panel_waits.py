"""The panels whose CTAs wait for one another: the register panel of a thread-block cluster
(pushes into the peers' shared memory) and the cooperative grid panel (published candidates),
here forced on small fronts.  A limit of 1 ns, far below a round trip, runs out on the first
waits: the panel reports it (bit 2 of the status), leaves interchanges inside the front, and the
device goes on working.  With the default limit the same fronts factor: FP32 bit for bit as on the
CPU, FP64 to the same pivots and the same first panel.
"""
import numpy as np
import pytest

from test_gpu_front_lu import check, factor, reference

pytestmark = pytest.mark.gpu

# rows, eliminated rows, fronts, on the grid: clusters of 2 (FP64) to 16 CTAs, grids of 1 to 66
CASES = [(1100, 64, 1, 0), (2100, 33, 1, 0), (4200, 33, 1, 0), (40, 33, 2, 1), (300, 64, 3, 1), (2100, 33, 1, 1)]


@pytest.mark.parametrize("T", [np.float32, np.float64])
@pytest.mark.parametrize("m,k,nf,grid", CASES)
def test_wait_and_result(m, k, nf, grid, T):
    rng = np.random.default_rng([m, k])
    A = rng.standard_normal((nf, m, m)).astype(T)
    got, piv, perm, st = factor(A, k, grid, wait_ns=1)
    if m > 40:  # a grid of one or two CTAs may find its peers' words at the first poll
        assert st & 2
    assert np.all(piv >= 0) and np.all(piv < k)
    got, piv, perm, st = factor(A, k, grid)
    assert st == 0
    if T == np.float32:
        check(A, k, got, piv, perm, {0, nf - 1}, np.array([k, m - 1]))
        return
    for f in {0, nf - 1}:
        ref, rp = reference(A[f], k, np.zeros(0, int))
        assert np.array_equal(piv[f], rp)
        assert np.array_equal(got[f][:, :32], ref[:, :32])
