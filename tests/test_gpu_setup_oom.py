"""A set-up that runs out of device memory gives back what it had allocated: a group of 20 problems
of 256^2 with eight right-hand sides and 1000 Krylov vectors each asks for 2 x 168 GB of basis."""
import pytest

pytestmark = pytest.mark.gpu


def test_failed_setup_frees_its_memory():
    import torch

    from paper_1409_0297_gb300 import binding as B

    torch.cuda.empty_cache()
    B.Solver(2, 64, 4, 414.5, restart=2, setup_route=1).close()  # the library's own start-up
    free = torch.cuda.mem_get_info()[0]
    if free > 330e9:
        pytest.skip("the request fits this GPU")
    with pytest.raises(B.SpError) as e:
        B.Solver(2, 256, 8, [414.5] * 20, prec=B.SP_PREC_FP32, restart=1000, max_rhs=8, setup_route=1)
    assert e.value.status == B.SP_ERR_OOM
    assert abs(torch.cuda.mem_get_info()[0] - free) < 1e9
