"""Front panels in every form of the panel factorisation: one warp, one CTA, clusters of 2
to 16 CTAs, and (FP64, 3D 48^3) the grid of CTAs beyond them.

The FP64 and the FP32 preconditioner factor the same fronts through different panel shapes
(rows per thread, CTAs per front).  Both solves run to a true residual of 1e-12; the
workloads here amplify a residual at most about 240-fold in the solution (measured with
the oracle at 512^2), so two right solutions agree within 2 x 240 x 1e-12 < 1e-9.
"""
import numpy as np
import pytest

import synthetic_media as sm

pytestmark = pytest.mark.gpu

# tallest fronts (rows of the first panels): 2D 4 n - 4 at the root, 3D as noted
GRIDS = [(2, 24, 3), (2, 96, 6), (2, 192, 6), (2, 384, 12), (3, 16, 4), (3, 32, 4), (3, 48, 6)]


@pytest.mark.parametrize("d,n,b", GRIDS)
def test_fp32_and_fp64_panels_give_one_solution(d, n, b):
    import torch

    from paper_1409_0297_gb300 import binding as B

    c = sm.grf_velocity(d, n, 0.05 if d == 2 else 0.08, 1000 + n)
    f = torch.from_numpy(sm.random_gaussian_source(d, n, 2000 + n)).cuda()
    s, q = B.sp_medium_helmholtz(d, n, 2 * np.pi * n / 8, c)
    q = torch.from_numpy(q).cuda()
    u = {}
    for prec in (B.SP_PREC_FP64, B.SP_PREC_FP32):
        S = B.Solver(d, n, b, s, prec=prec, tol=1e-12, setup_route=1 if d == 3 else 0)
        S.factor(q)
        u[prec] = torch.empty_like(f)
        info = S.solve(f, u[prec])
        S.close()
        assert info["true_relres"] <= 1e-12
    err = torch.linalg.norm(u[B.SP_PREC_FP32] - u[B.SP_PREC_FP64]) / torch.linalg.norm(u[B.SP_PREC_FP64])
    assert float(err) <= 1e-9
