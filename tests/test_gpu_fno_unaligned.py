"""Network inputs that do not start on a 16-byte boundary take plain loads and give the bits
of aligned ones (forward pass, loss and gradient)."""
import numpy as np
import pytest

import synthetic_media as sm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("act_fp32", [False, True])
@pytest.mark.parametrize("c_in,width,modes,hidden,batch", [(3, 8, 6, 48, 1), (5, 30, 15, 100, 9)])
def test_unaligned_input(act_fp32, c_in, width, modes, hidden, batch):
    import torch

    from paper_1409_0297_gb300 import binding as B

    n = 64
    p = sm.fno_initial_params(c_in, width, modes, 2, hidden, 2)
    F = B.Fno(n, p, c_in=c_in, width=width, modes=modes, layers=2, hidden=hidden, batch_max=batch,
              act_fp32=act_fp32)
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randn(batch * c_in * n * n, generator=g, device="cuda")
    t = torch.randn(batch * 2 * n * n, generator=g, device="cuda")
    out = []
    for off in (0, 1):
        buf = torch.empty(x.numel() + 4, device="cuda")
        xs = buf[off:off + x.numel()]
        xs.copy_(x)
        assert (xs.data_ptr() % 16 == 0) == (off == 0)
        y = torch.empty(batch * 2 * n * n, device="cuda")
        F.forward(xs, y, batch)
        loss, grad = F.gradient(xs, t, batch)
        out.append((y.cpu().numpy(), loss, grad))
    F.close()
    assert np.array_equal(out[0][0], out[1][0])
    assert out[0][1] == out[1][1]
    assert np.array_equal(out[0][2], out[1][2])
