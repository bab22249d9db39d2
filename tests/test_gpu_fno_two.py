"""Two networks of different size alive at once: a small one made later leaves the launches of the
large one as they were (loss and gradient bit for bit those of the large one alone)."""
import numpy as np
import pytest

import synthetic_media as sm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,batch", [(32, 16), (32, 256), (8, 64)])
def test_small_network_beside_a_large_one(width, batch):
    import torch

    from paper_1409_0297_gb300 import binding as B

    n = 64
    net = lambda w, b: B.Fno(n, sm.fno_initial_params(3, w, 4, 1, 16, 2), c_in=3, width=w, modes=4, layers=1,
                             hidden=16, batch_max=b)
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn(batch * 3 * n * n, generator=g, device="cuda")
    t = torch.randn(batch * 2 * n * n, generator=g, device="cuda")
    large = net(width, batch)
    loss, grad = large.gradient(x, t, batch)
    small = net(2, 1)
    again = large.gradient(x, t, batch)
    small.gradient(x, t, 1)
    last = large.gradient(x, t, batch)
    for got in (again, last):
        assert got[0] == loss and np.array_equal(got[1], grad)
    small.close()
    large.close()
