"""Register levels of few samples run on twice the lanes: the same samples from
a batch just below and just above the size where that ends (coupled and plain,
one and four test functions) are equal, masses and moment sums too."""
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


def _run(ctx, dk, level, mc, count):
    import torch
    sums = torch.zeros(dk.sums_len(ctx.n_quant), dtype=torch.float64, device="cuda")
    samp = torch.zeros(count, dk.sample_stride(ctx.n_obs), dtype=torch.float64, device="cuda")
    ctx.run_level_dev(level, int(mc), 7, count, 5, sums.data_ptr(), samp.data_ptr(),
                      torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return sums.cpu().numpy(), samp.cpu().numpy()


@pytest.mark.parametrize("four", [False, True])
@pytest.mark.parametrize("n0,level,mc,most", [(16, 0, False, 912), (16, 0, True, 912), (8, 1, False, 912),
                                              (16, 1, False, 456), (16, 1, True, 456)])
def test_few_sample_shape_gives_the_same_samples(dk, n0, level, mc, most, four):
    """The same integer paths and the same FP32 projection sums; only FP64 sums
    over lanes run in another order (32 lanes to 128: 7 roundings of 2^-53 of the
    partial sums' size, which is at most 10^3 of their total's)."""
    wl = W.get("mlmc16_256").with_(n0=n0, L_max=max(level, 1), T=0.004)
    if four:
        wl = wl.with_(observables=W.get("large32_1024").observables, products=True)
    with dk.Context.from_workload(wl) as ctx:
        big_sums, big = _run(ctx, dk, level, mc, most + 1)
        for count in (1, 5, most):
            sums, samp = _run(ctx, dk, level, mc, count)
            scale = np.sqrt(np.mean(big ** 2, axis=0))
            assert np.max(np.abs(samp - big[:count]) / np.maximum(scale, 1e-300)) <= 1e3 * 7 * 2.0 ** -53
            assert int(sums[0]) == count and sums[1] == 0.0
            dp = wl.N * (samp[:, 0] ** 2 - (samp[:, ctx.n_obs] ** 2 if level > 0 and not mc else 0.0))
            np.testing.assert_allclose(sums[2], dp.sum(), rtol=1e-9, atol=1e-9 * np.abs(dp).sum())


@pytest.mark.parametrize("level,mosts", [(2, (456,)), (3, (304, 608)), (4, (152,))])
@pytest.mark.parametrize("mc", [False, True])
def test_few_samples_of_the_fluctuation_state(dk, level, mosts, mc):
    """16^2, 32^2 and 64^2 about the noise-free path: the shapes for few samples on
    both sides of each size where one ends, by the same measure."""
    wl = W.get("paper_reg").with_(L_max=level)
    with dk.Context.from_workload(wl) as ctx:
        assert ctx.level_info(level).n == 4 << level
        _, big = _run(ctx, dk, level, mc, 700)
        scale = np.sqrt(np.mean(big ** 2, axis=0))
        for most in mosts:
            for count in (most, most + 1):
                sums, samp = _run(ctx, dk, level, mc, count)
                assert np.max(np.abs(samp - big[:count]) / np.maximum(scale, 1e-300)) <= 1e3 * 7 * 2.0 ** -53
                assert int(sums[0]) == count and sums[1] == 0.0


@pytest.mark.parametrize("name,mc", [("fourier6_54", False), ("fourier6_54", True), ("paper_reg_fourier", False)])
def test_few_samples_of_the_18_grid(dk, name, mc):
    """18^2 Fourier level, absolute and fluctuation state: one and two rows of cells
    per thread give the same samples, up to the same order of FP64 sums."""
    wl = W.get(name).with_(L_max=1)
    with dk.Context.from_workload(wl) as ctx:
        assert ctx.level_info(1).n == 18
        big_sums, big = _run(ctx, dk, 1, mc, 1217)
        assert int(big_sums[0]) == 1217 and big_sums[1] == 0.0
        for count in (1, 1216):
            sums, samp = _run(ctx, dk, 1, mc, count)
            scale = np.sqrt(np.mean(big ** 2, axis=0))
            assert np.max(np.abs(samp - big[:count]) / np.maximum(scale, 1e-300)) <= 1e3 * 7 * 2.0 ** -53
            assert int(sums[0]) == count and sums[1] == 0.0
