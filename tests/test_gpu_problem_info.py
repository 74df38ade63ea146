"""acs_problem_info describes the launch that a solve makes: one cluster of 8 or 16 CTAs
of 512 threads for a small problem with the cached operator, else the whole grid."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2103_00736_gb300 import capi, instances as I  # noqa: E402


@pytest.mark.parametrize("m,projection,small", [(100, capi.PROJ_DENSE, True), (100, capi.PROJ_CG, False),
                                                (600, capi.PROJ_DENSE, False)])
def test_launch(m, projection, small):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    with capi.Solver(I.bernoulli_lp(m, m, 2 * m), projection=projection) as s:
        info = capi.acs_problem_info(s.h)
        s.solve(tol=0.0, max_iter=1)
        torch.cuda.synchronize()
    assert info["grid32"] == sms
    if small:
        assert info["grid64"] in (8, 16) and info["threads"] == 512
    else:
        assert info["grid64"] == sms and info["threads"] == 1024
