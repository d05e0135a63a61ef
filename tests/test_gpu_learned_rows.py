"""Learned level: the rows that a batch of 4864 (64-column tiles) and one of 4865 (256
columns) have in common are equal, bit for bit: the same FP32 sums in the same
order from both tile widths."""
import importlib.util
import os

import numpy as np
import pytest

from oracle import surrogate as sg
from paper_2311_08872_gb300 import workloads as W

pytestmark = pytest.mark.gpu

_spec = importlib.util.spec_from_file_location(
    "surrogate_reference", os.path.join(os.path.dirname(__file__), "test_gpu_surrogate.py"))
ref = importlib.util.module_from_spec(_spec)
_spec.loader.exec_module(ref)
dk = ref.dk


def test_rows_do_not_depend_on_the_tile_width(dk):
    wl = W.get("mlmc16_256").with_(L_max=1)
    rng = np.random.default_rng(9)
    theta = rng.normal(0, 0.08, size=sg.mlp_param_count(1)).astype(np.float32)
    X = rng.normal(size=(4865, 64)).astype(np.float32)
    with dk.Context.from_workload(wl) as ctx:
        ctx.surrogate_init(0)
        ctx.surrogate_params(theta)
        narrow, wide = ctx.surrogate_forward(X[:4864]), ctx.surrogate_forward(X)
    assert np.isfinite(wide).all() and np.ptp(wide) > 0
    np.testing.assert_array_equal(narrow, wide[:4864])
