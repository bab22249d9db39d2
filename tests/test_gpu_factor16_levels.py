"""Which levels keep the FP16 copy of the factor (sp_opts.factor_storage = 1): those whose fronts
do not fill the GPU (fewer than 304, two to each of 152 SMs).  Levels of many fronts read FP32,
whether they are swept by fused launches or, for their few rows, by launch chains."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,n,b", [(2, 128, 4), (2, 192, 6), (2, 256, 8), (2, 192, 12), (3, 32, 4), (3, 24, 3)])
def test_levels_of_many_fronts_stay_fp32(d, n, b):
    import torch

    from paper_1409_0297_gb300 import binding as B

    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the line is two fronts to each of 152 SMs")
    S = B.Solver(d, n, b, 414.5, prec=B.SP_PREC_FP32, factor_storage=1, setup_route=1, restart=2)
    got = B.sp_costs(S.ctx)["apply_bytes"]
    S.close()
    want = sum(nf * (k * k + 2.0 * k * (m - k)) * (4 if nf >= 304 else 2)
               for nf, k, m in B.sp_front_sizes(d, n, b))
    assert got == want
