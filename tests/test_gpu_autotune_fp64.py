"""sp_opts.autotune in FP64: the digit products have one tile, so every level reports 64 (and the
same for the block inverses of the levels that keep them)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n,b", [(2, 128, 8), (2, 96, 6), (3, 16, 4)])
def test_one_tile(d, n, b):
    from paper_1409_0297_gb300 import binding as B

    for _ in range(3):  # timings would differ from one set-up to the next
        S = B.Solver(d, n, b, 414.5, prec=B.SP_PREC_FP64, autotune=True, setup_route=1, restart=2)
        for level, (nf, k, m) in enumerate(B.sp_front_sizes(d, n, b)):
            t = B.sp_tuning(S.ctx, level)
            assert t["gemm_tile"] == 64
            assert t["gen_tile"] == (64 if nf < 152 else 0)
        S.close()
