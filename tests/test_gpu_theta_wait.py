"""Failure detection of the 128^2 theta-scheme cluster kernel without a fault: the
first CTA of every cluster stops before a fine step, its neighbours' waits
(limited to 4096 polls) run out, the kernel records the timeout and finishes, the
call returns MLMC_DK_ERR_TIMEOUT, and the same context then runs the same samples
as before."""
import numpy as np
import pytest

from paper_2311_08872_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dk():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2311_08872_gb300 import build as libbuild
    libbuild.build()
    from paper_2311_08872_gb300 import mlmc_dk
    return mlmc_dk


def _samples(ctx, dk, count):
    import torch
    sums = torch.zeros(dk.sums_len(1), dtype=torch.float64, device="cuda")
    samp = torch.zeros(count, dk.sample_stride(1), dtype=torch.float64, device="cuda")
    ctx.run_level_dev(3, 0, 0, count, 9, sums.data_ptr(), samp.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return sums.cpu().numpy(), samp.cpu().numpy()


# (both builds, few samples and many; first, inner and last step; a coarse step's end)
@pytest.mark.parametrize("count,step", [(1, 0), (1, 7), (3, 15), (40, 0), (100, 3), (160, 8)])
def test_bounded_wait_reports_timeout(dk, count, step):
    wl = W.get("theta16_128").with_(T=0.001)
    with dk.Context.from_workload(wl) as ctx:
        assert ctx.level_info(3).cluster == 4 and ctx.level_info(3).M >= 16
        before = _samples(ctx, dk, 40)
        assert ctx.theta_wait_test(3, count, 4096, step) == dk.ERR_TIMEOUT
        assert ctx.run_level(3, 2, 9)[0].n == 2          # the error does not stick
        after = _samples(ctx, dk, 40)
    np.testing.assert_array_equal(before[1], after[1])
    np.testing.assert_array_equal(before[0], after[0])


def test_wait_test_arguments(dk):
    wl = W.get("theta16_128").with_(T=0.001)
    with dk.Context.from_workload(wl) as ctx:
        assert ctx.theta_wait_test(2, 1, 4096, 0) == dk.ERR_UNSUPPORTED    # 64^2: no cluster
        assert ctx.theta_wait_test(3, 1, 0, 0) == dk.ERR_INVALID
        assert ctx.theta_wait_test(3, 0, 4096, 0) == dk.ERR_INVALID
        assert ctx.theta_wait_test(3, 1, 4096, -1) == dk.ERR_INVALID
