"""Lines of the FFT passes at the edges of their launch shapes: two and four points, one step,
a radix 3 behind one or two steps, and lines of 2048 points (two butterflies per thread).

Against numpy's transform of the same operator: both are FP64 transforms whose relative error
grows like eps log2 N; 1e-12 of the result leaves a factor of 100 over eps log2(2048^2) times
the operator's norm here (q at most 1, symbol at most 1 / (s gap) with s = 4 pi^2 10.5).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n,b", [(2, 8, 2), (2, 12, 3), (2, 24, 3), (2, 48, 6), (2, 96, 6),
                                   (2, 1536, 12), (2, 2048, 32), (3, 8, 2), (3, 12, 3), (3, 24, 3)])
def test_operator_against_numpy(d, n, b):
    import torch

    from paper_1409_0297_gb300 import binding as B

    s = 4 * np.pi ** 2 * 10.5
    rng = np.random.default_rng([d, n])
    x = rng.standard_normal(n ** d) + 1j * rng.standard_normal(n ** d)
    q = rng.uniform(-1.0, 1.0, n ** d)
    S = B.Solver(d, n, b, s, prec=B.SP_PREC_FP32, restart=2, setup_route=1)
    qd = torch.from_numpy(q).cuda()
    S.factor(qd)
    xd = torch.from_numpy(x).cuda()
    w, g = torch.empty_like(xd), torch.empty_like(xd)
    S.matvec(xd, w)
    S.green(xd, g)
    k = np.fft.fftfreq(n, d=1.0 / n)
    k2 = sum(np.square(a) for a in np.meshgrid(*([k] * d), indexing="ij"))
    sym = 1.0 / (4 * np.pi ** 2 * k2 - s)
    ref = lambda v: np.fft.ifftn(np.fft.fftn(v.reshape((n,) * d)) * sym).ravel()
    for got, want in ((w, x + ref(q * x)), (g, ref(x))):
        got = got.cpu().numpy()
        assert np.linalg.norm(got - want) <= 1e-12 * np.linalg.norm(want)
    S.close()
