"""Register shapes with two builds (registers per thread) run the same arithmetic:
the same samples from batches on both sides of every size where the build changes,
and sums over the slots that were launched, also where a build keeps fewer samples
resident than the other (several passes of a smaller grid) and where the static
scratch limits the grid further."""
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


def _run(ctx, dk, level, mc, count, static=False):
    import torch
    st = torch.cuda.current_stream().cuda_stream
    sums = torch.full((dk.sums_len(ctx.n_quant),), float("nan"), dtype=torch.float64, device="cuda")
    samp = torch.full((count, dk.sample_stride(ctx.n_obs)), float("nan"), dtype=torch.float64, device="cuda")
    if static:
        ctx.run_level_static(level, int(mc), 7, count, 5, sums.data_ptr(), samp.data_ptr(), 0, st)
    else:
        ctx.run_level_dev(level, int(mc), 7, count, 5, sums.data_ptr(), samp.data_ptr(), st)
    torch.cuda.synchronize()
    return sums.cpu().numpy(), samp.cpu().numpy()


FL = "paper_reg"        # N = 2e9: fluctuation state


@pytest.mark.parametrize("name,n0,level,variant,mc,counts", [
    (FL, 4, 4, 0, False, (152, 153, 305, 418, 419, 456, 457, 760)),
    (FL, 4, 4, 0, True, (152, 153, 456)),
    (FL, 4, 3, 0, False, (608, 609, 1216, 1672, 1673, 1824, 1825, 4256, 5472)),
    (FL, 4, 3, 0, True, (912, 913, 1216, 1217, 2128, 2129, 2432, 2433)),
    (FL, 4, 1, 0, False, (4864, 4865, 6081)),
    (FL, 4, 1, 0, True, (4864, 4865, 6081)),
    ("mlmc16_256", 16, 0, 2, True, (912, 913, 1824, 3648, 3649)),
    ("mlmc16_256", 8, 1, 2, False, (912, 913, 1824, 3648, 3649)),
    ("mlmc16_256", 16, 1, 1, False, (456, 457, 608, 609)),
    ("mlmc16_256", 16, 1, 1, True, (456, 457, 608, 609)),
    ("mlmc16_256", 16, 1, 2, False, (456, 457, 608, 609)),
    ("mlmc16_256", 16, 1, 2, True, (456, 457, 608, 609)),
])
def test_both_builds_give_the_same_samples(dk, name, n0, level, variant, mc, counts):
    """Integer paths and per-lane FP32 sums are the same; only FP64 sums over lanes and
    slots run in another order (at most 2^13 terms: 13 roundings of 2^-53 of the partial
    sums' size, which is at most 10^3 of their total's)."""
    wl = W.get(name)
    wl = wl.with_(L_max=max(level, 1)) if name == FL else wl.with_(n0=n0, L_max=max(level, 1), T=0.004)
    with dk.Context.from_workload(wl) as ctx:
        assert ctx.level_info(level).n == wl.n0 << level
        ctx.set_variant(level, level > 0 and not mc, variant)
        _, big = _run(ctx, dk, level, mc, max(counts))
        assert np.isfinite(big).all()
        scale = np.maximum(np.sqrt(np.mean(big ** 2, axis=0)), 1e-300)
        for count in counts:
            for static in (False, True):
                sums, samp = _run(ctx, dk, level, mc, count, static)
                assert np.max(np.abs(samp - big[:count]) / scale) <= 1e3 * 13 * 2.0 ** -53
                assert int(sums[0]) == count and sums[1] == 0.0
                coarse = samp[:, ctx.n_obs] if level > 0 and not mc else 0.0
                dp = wl.N * (samp[:, 0] ** 2 - coarse ** 2)
                np.testing.assert_allclose(sums[2], dp.sum(), rtol=1e-9, atol=1e-9 * np.abs(dp).sum())


@pytest.mark.parametrize("mc", [False, True])
def test_both_builds_of_the_16_grid_theta_level(dk, mc):
    """16^2 theta level: both builds run the same operations on every cell; the FP64
    sums over lanes too."""
    wl = W.get("theta16_128").with_(n0=8, L_max=1, T=0.02)
    with dk.Context.from_workload(wl) as ctx:
        assert ctx.level_info(1).n == 16 and ctx.level_info(1).theta == 1
        _, big = _run(ctx, dk, 1, mc, 4000)
        for count in (1, 1825, 2128, 2129, 3040, 3041, 3648, 3649, 4000):
            for static in (False, True):
                sums, samp = _run(ctx, dk, 1, mc, count, static)
                np.testing.assert_array_equal(samp, big[:count])
                assert int(sums[0]) == count and sums[1] == 0.0
                dp = wl.N * (samp[:, 0] ** 2 - (0.0 if mc else samp[:, 1] ** 2))
                np.testing.assert_allclose(sums[2], dp.sum(), rtol=1e-9, atol=1e-9 * np.abs(dp).sum())


@pytest.mark.parametrize("mc", [False, True])
def test_both_builds_of_the_54_grid_fourier_level(dk, mc):
    """54^2 Fourier level with the fluctuation state: few samples run on one row of
    cells per thread.  Integer paths are the same; the FP64 sums over threads (486 of
    them: 9 levels, partial sums at most 10^3 of their total) run in another order."""
    wl = W.get("paper_reg_fourier")
    with dk.Context.from_workload(wl) as ctx:
        assert ctx.level_info(2).n == 54 and ctx.level_info(2).fluct == 1
        _, big = _run(ctx, dk, 2, mc, 305)
        scale = np.maximum(np.sqrt(np.mean(big ** 2, axis=0)), 1e-300)
        for count in (1, 152, 153, 305):
            for static in (False, True):
                sums, samp = _run(ctx, dk, 2, mc, count, static)
                assert np.max(np.abs(samp - big[:count]) / scale) <= 1e3 * 9 * 2.0 ** -53
                assert int(sums[0]) == count and sums[1] == 0.0


@pytest.mark.parametrize("mc", [False, True])
def test_three_builds_of_the_32_grid_theta_level(dk, mc):
    """32^2 theta level: 2 x 2, 4 x 2 and 4 x 4 blocks per thread run the same operations
    on every cell, up to the order of the FP64 sums over threads (256: 8 levels)."""
    wl = W.get("theta16_128").with_(L_max=1, T=0.005)
    with dk.Context.from_workload(wl) as ctx:
        assert ctx.level_info(1).n == 32 and ctx.level_info(1).theta == 1
        _, big = _run(ctx, dk, 1, mc, 900)
        scale = np.maximum(np.sqrt(np.mean(big ** 2, axis=0)), 1e-300)
        for count in (1, 304, 305, 608, 609, 900):
            for static in (False, True):
                sums, samp = _run(ctx, dk, 1, mc, count, static)
                assert np.max(np.abs(samp - big[:count]) / scale) <= 1e3 * 8 * 2.0 ** -53
                assert int(sums[0]) == count and sums[1] == 0.0
