"""Theta-scheme solve at the ends of its range of Chebyshev steps (one step, two,
and dozens at a large tau/h^2) on every layout of the kernel: a warp or less per
sample, several warps, and a cluster of CTAs."""
import importlib.util
import os

import numpy as np
import pytest

from paper_2311_08872_gb300 import workloads as W

pytestmark = pytest.mark.gpu

_spec = importlib.util.spec_from_file_location(
    "theta_reference", os.path.join(os.path.dirname(__file__), "test_gpu_theta.py"))
ref = importlib.util.module_from_spec(_spec)
_spec.loader.exec_module(ref)
dk = ref.dk


@pytest.mark.parametrize("b0,mu,steps", [(1e-9, 0.4, (1, 1)), (1e-4, 0.4, (2, 3)), (1.0, 6.0, (40, 64))])
@pytest.mark.parametrize("level,count,T", [(0, 9, 0.02), (1, 5, 0.02), (2, 3, 0.02), (3, 2, 0.005)])
def test_chebyshev_step_range(dk, b0, mu, steps, level, count, T):
    wl = W.get("theta16_64").with_(b0=b0, mu=mu, L_max=3, T=T)
    seed, first = 91 + level, 1
    with dk.Context.from_workload(wl) as ctx:
        info = ctx.level_info(level)
        assert info.n == 16 << level and (T < 0.02 or steps[0] <= info.cheb_steps <= steps[1])
        sums, samp = ref._gpu(ctx, dk, level, 0, first, count, seed)
    r, ybf, ybc = ref._oracle(wl, level, 0, first, count, seed)
    ref._parity(samp[:, :1] + ybf[None, :], r["Y_f"], ybf, f"b0 {b0} level {level} fine")
    if ybc is not None:
        ref._parity(samp[:, 1:2] + ybc[None, :], r["Y_c"], ybc, f"b0 {b0} level {level} coarse")
    assert int(sums[0]) == count and sums[1] == 0.0
    assert np.isfinite(samp).all()


@pytest.mark.parametrize("level,held,mc", [(1, 304, False), (1, 304, True), (2, 152, False), (2, 152, True), (3, 36, False), (3, 36, True)])
def test_batches_on_both_sides_of_the_residency_rule(dk, level, held, mc):
    """The two builds of a grid size (few and many resident samples) run the same
    operations on every cell: the same samples from a batch of `held` and of many
    more (several passes of the persistent grid), up to the order of the FP64 sums
    over threads (log2 of 1024 threads roundings of 2^-53 of the partial sums' size,
    at most 10^3 of their total's)."""
    wl = W.get("theta16_64").with_(L_max=3, T=0.005)
    with dk.Context.from_workload(wl) as ctx:
        assert ctx.level_info(level).n == 16 << level
        _, few = ref._gpu(ctx, dk, level, int(mc), 3, held, 17)
        for count in (held + 1, 5 * held + 3):
            sums, many = ref._gpu(ctx, dk, level, int(mc), 3, count, 17)
            assert int(sums[0]) == count and sums[1] == 0.0
            scale = np.sqrt(np.mean(many ** 2, axis=0))
            err = np.abs(few - many[:held]) / np.maximum(scale, 1e-300)
            assert err.max() <= 1e3 * 10 * 2.0 ** -53
