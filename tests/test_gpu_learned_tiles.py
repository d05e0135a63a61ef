"""Learned level: batch sizes at the edges of the tensor-core tiles and of the
launch rule (rows of 128, one or two CTAs' worth of columns), and of the
batch sums (256 rows per pass, ragged and single-row batches)."""
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


def _exact_network(rng, outputs):
    """Parameters for which every stored value is exact: two features of weight +-1
    per unit of the first layer, signed permutations after it, integer biases, and
    one output a unit.  With integer features all activations are small integers
    and every entry of the activations' gradients is one product, so masks and
    BF16 values are those of the reference and only the sums over the batch round."""
    W1 = np.zeros((256, 64))
    for i in range(256):
        W1[i, rng.choice(64, 2, replace=False)] = rng.choice([-1.0, 1.0], 2)
    layers = [(W1, rng.integers(0, 3, 256))]
    for _ in range(2):
        P = np.zeros((256, 256))
        P[np.arange(256), rng.permutation(256)] = rng.choice([1.0, 1.0, 1.0, -1.0], 256)
        layers.append((P, rng.integers(0, 3, 256)))
    W4 = np.zeros((outputs, 256))
    W4[rng.integers(0, outputs, 256), np.arange(256)] = rng.choice([-1.0, 1.0], 256)
    layers.append((W4, rng.integers(-3, 3, outputs)))
    return np.concatenate([np.concatenate([W.reshape(-1), np.asarray(b, float)]) for W, b in layers]).astype(np.float32)


@pytest.mark.parametrize("outputs,B", [(1, 1), (1, 127), (1, 128), (1, 129), (4, 255), (1, 257), (4, 1000), (1, 4096)])
def test_gradient_at_batch_edges(dk, outputs, B):
    """Each gradient entry is a sum over the batch of B exact products: in FP32, in
    any order, off by at most B 2^-24 of the sum of their magnitudes; the output
    gradient d = 2 (y - t) / B is itself rounded by 2^-24 and stored in BF16 by
    both sides (a tie or a neighbour's rounding cannot differ: y - t is an integer)."""
    wl = W.get("mlmc16_256" if outputs == 1 else "large32_1024").with_(L_max=1)
    rng = np.random.default_rng(B)
    theta = _exact_network(rng, outputs)
    X = rng.integers(-2, 3, size=(B, 64)).astype(np.float32)
    T = rng.integers(-20, 20, size=B if outputs == 1 else (B, outputs)).astype(np.float32)
    _, loss, grad = ref._bf16_network(theta, X, T)
    # the sums of magnitudes: the same network's products without their signs
    (W1, b1), (W2, b2), (W3, b3), (W4, b4) = sg.mlp_unpack(theta.astype(np.float64), outputs)
    H1 = np.maximum(X.astype(np.float64) @ W1.T + b1, 0)
    H2 = np.maximum(H1 @ W2.T + b2, 0)
    H3 = np.maximum(H2 @ W3.T + b3, 0)
    assert max(H1.max(), H2.max(), H3.max()) <= 256
    d = np.abs(2.0 * (H3 @ W4.T + b4 - T.reshape(B, outputs)) / B)
    D3 = (d @ np.abs(W4)) * (H3 > 0)
    D2 = (D3 @ np.abs(W3)) * (H2 > 0)
    D1 = (D2 @ np.abs(W2)) * (H1 > 0)
    mag = np.concatenate([v.reshape(-1) for v in (
        D1.T @ np.abs(X), D1.sum(0), D2.T @ H1, D2.sum(0), D3.T @ H2, D3.sum(0), d.T @ H3, d.sum(0))])
    with dk.Context.from_workload(wl) as ctx:
        ctx.surrogate_init(0)
        ctx.surrogate_params(theta)
        got_loss, got = ctx.surrogate_loss_grad(X, T)
    assert abs(got_loss - loss) <= 1e-12 * loss
    # |d| in BF16 is at most 1 + 2^-8 of |d|
    bound = (B + 2) * 2.0 ** -24 * 1.01 * mag
    assert got.shape == grad.shape
    worst = np.abs(got - grad) - bound
    assert worst.max() <= 0, (int(worst.argmax()), float(worst.max()))


@pytest.mark.parametrize("n", [1, 4864, 4865])
def test_forward_on_both_sides_of_the_tile_rule(dk, n):
    """A row's result does not depend on the tile it is in: the same FP32 sums in
    the same order from 64- and 256-column tiles."""
    wl = W.get("mlmc16_256").with_(L_max=1)
    rng = np.random.default_rng(8)
    theta = rng.normal(0, 0.08, size=sg.mlp_param_count(1)).astype(np.float32)
    X = rng.normal(size=(4865, 64)).astype(np.float32)
    with dk.Context.from_workload(wl) as ctx:
        ctx.surrogate_init(0)
        ctx.surrogate_params(theta)
        y = ctx.surrogate_forward(X[:n])
        small = ctx.surrogate_forward(X[n - 1:n])
    np.testing.assert_array_equal(y[n - 1:n], small)
