"""Range of the theta-scheme's face fluxes.  The coarse step's raw face flux (the
diffusion flux plus the two noise transfers) may leave 32 bits as long as the
corrected flux and the state stay in range: such a sample is valid and agrees with
the exact solve."""
import math

import numpy as np
import pytest

import oracle

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


A = 1.6          # initial density of the fine path; the coarse one jumps between A and -A
MU = 9.95        # tau / h^2: the flux across a jump is 0.995 x 2^31 in fixed point
S = 27           # 2^S (2 A + 12 standard deviations) < 2^29


def _setup(n0):
    """One coarse step on n0^2, four fine steps on (2 n0)^2."""
    N = 1e5 * (n0 / 16) ** 2
    levels = oracle.level_table(1.0, n0, 1, MU / n0 ** 2, MU, 1)
    rho_c = np.where(np.arange(n0)[:, None] < n0 // 2, A, -A) * np.ones((n0, n0))
    rho0 = [rho_c, np.full((2 * n0, 2 * n0), A)]
    phi = []
    for l in range(2):
        x = np.arange(levels[l].n) * levels[l].h
        phi.append([np.cos(2 * math.pi * x)[:, None] * np.ones((1, levels[l].n))])
    return N, levels, rho0, phi


def _raw_flux(n0, N, levels, rho_c, seed, sample):
    """Largest raw face flux of the coarse step in units of 2^-S (FP64)."""
    n, h, tau = n0, levels[0].h, levels[0].tau
    Z = sum(oracle.normals(seed, 1, 0, sample, m, 2 * n) for m in range(4))
    Z = Z.reshape(n, 2, n, 2, 2).sum((1, 3)) / 4
    c = math.sqrt(tau / N) / (2 * h * h)
    worst = 0.0
    for ax in range(2):
        G = c * np.sqrt(np.maximum(rho_c, 0)) * Z[..., ax]
        F = tau / (2 * h * h) * (np.roll(rho_c, -1, ax) - rho_c) + G + np.roll(G, -1, ax)
        worst = max(worst, np.abs(F).max())
    return worst * 2.0 ** S


@pytest.mark.parametrize("n0,count", [(8, 9), (16, 8), (16, 320), (32, 6), (32, 160), (64, 4), (64, 40)])
def test_coarse_raw_flux_beyond_32_bits(dk, n0, count):
    """The correction's FP32 error is at most K (<= 64) roundings of 2^-24 of the
    largest flux (2^31 2^-S), and enters the projection on cos as differences of two
    faces: 2 K 2^-24 2^(31 - S) bounds the error of Y."""
    import torch
    N, levels, rho0, phi = _setup(n0)
    seed = 5
    checked = range(min(count, 4))
    assert max(_raw_flux(n0, N, levels, rho0[0], seed, s) for s in checked) > 2.0 ** 31
    with dk.Context(1.0, n0, 1, levels[0].tau, MU, N, rho0, phi, M0=1, theta_b0=1.0) as ctx:
        info = ctx.level_info(1)
        assert info.theta == 1 and info.n == 2 * n0 and info.M == 4
        sums = torch.zeros(dk.sums_len(1), dtype=torch.float64, device="cuda")
        samp = torch.zeros(count, dk.sample_stride(1), dtype=torch.float64, device="cuda")
        err = torch.zeros(1, dtype=torch.int32, device="cuda")
        ctx.run_level_static(1, 0, 0, count, seed, sums.data_ptr(), samp.data_ptr(), err.data_ptr(),
                             torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        assert int(err.item()) == 0
        assert ctx.run_level(1, count, seed)[0].n == count
        ybar = float(info.ybar_c[0])
    samp, sums = samp.cpu().numpy(), sums.cpu().numpy()
    assert sums[0] == count and sums[1] == 0.0
    ol = oracle.level_inputs(1.0, levels, N, rho0, phi, 1, True, b0=1.0)
    r = oracle.run_samples(ol, seed, checked, True, stream=0)
    bound = 2 * 64 * 2.0 ** -24 * 2.0 ** (31 - S)
    assert np.abs(samp[:len(checked), 1] + ybar - r["Y_c"][:, 0]).max() <= bound
