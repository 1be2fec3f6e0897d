"""The proposal network's training kernels at the shapes where their tiles and sums can go
wrong: batches around 128 and 256 rows (chunks of rows, padding), embedding widths that
are no multiple of 32 and above it, one row, many rows of one pair, and a batch large
enough to split the weight gradients' K.

Bars as in the training parity tests against the FP64 oracle: every gradient within 1e-2 of
its tensor's largest magnitude (operands are rounded to bf16 on both sides; FP32 against
FP64 accumulation), the first Adam step at most lr (1 + 1e-5) per element and opposite in
sign to a gradient that is not near zero."""
import numpy as np
import pytest

import synth
from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,H,B", [(6, 8, 128, 1), (7, 5, 128, 127), (9, 33, 128, 129), (12, 40, 256, 255),
                                     (20, 16, 128, 257), (6, 8, 128, 2100)])
def test_training_step_shapes(gpu, n, d, H, B):
    rng = np.random.default_rng(B + d)
    w = synth.mlp_init_weights(n, d, H, 3)
    w["b1"] = rng.normal(0, 0.1, H).astype(np.float32)
    w["b2"] = rng.normal(0, 0.1, H).astype(np.float32)
    P = n * (n - 1) // 2
    orders = synth.random_orders(n, B, 7)
    pairs = rng.integers(0, P, B).astype(np.uint32)
    pairs[: B // 3] = 2 % P                                     # one pair in a third of the rows
    alpha = rng.random(B).astype(np.float32)
    net = gpu.mlp_create(n, w, hidden=H, d=d, batch_cap=B, lr=1e-3)
    loss = gpu.mlp_loss_grad(net, orders, pairs, alpha)
    prm = omlp.MLPParams(*(np.asarray(w[k], np.float64) for k in gpu.MLP_TENSORS))
    ref_loss, ref = omlp.mlp_loss_grad(prm, orders, pairs.astype(np.int64), alpha.astype(np.float64))
    assert loss == pytest.approx(ref_loss, rel=1e-2)
    grads = {k: gpu.mlp_read(net, k, grad=True) for k in gpu.MLP_TENSORS}
    for k, g in grads.items():
        assert np.abs(g - ref[k]).max() <= 1e-2 * np.abs(ref[k]).max(), k
    untouched = np.setdiff1d(np.arange(P), pairs)
    assert not grads["W3"][untouched].any() and not grads["b3"][untouched].any()
    gpu.mlp_adam_step(net)
    for k, g in grads.items():
        step = gpu.mlp_read(net, k) - w[k]
        assert np.abs(step).max() <= 1e-3 * (1 + 1e-3) + 1e-6, k
        big = np.abs(g) > 1e-6
        assert (np.sign(step[big]) == -np.sign(g[big])).all(), k
    # the bf16 copies follow the weights: the forward of the stepped network
    new = omlp.MLPParams(*(np.asarray(gpu.mlp_read(net, k), np.float64) for k in gpu.MLP_TENSORS))
    logits, want = gpu.mlp_forward(net, orders), omlp.mlp_forward(new, orders)["logits"]
    assert np.abs(logits - want).max() <= 1e-2 * np.abs(want).max()
