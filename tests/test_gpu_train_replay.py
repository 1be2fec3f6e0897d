"""Training steps replayed from a captured graph (chains_step) against the same steps launched
one by one (chains_step_profiled): Adam's bias corrections belong to the step that runs, so
the weights must be the same bit for bit, also when calls are split and explicit Adam steps
come in between; and after steps without gradients in between, against Adam in FP64."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
TENSORS = ("E", "W1", "b1", "W2", "b2", "W3", "b3")


def _weights(gpu, net):
    return {x: gpu.mlp_read(net, x) for x in TENSORS}


@pytest.mark.parametrize("scan", ["full", "pruned"])
def test_replayed_training_equals_launched_training(gpu, scan):
    n, C = 9, 40
    rng = np.random.default_rng(2)
    t = gpu.table_from_scores(rng.normal(-100.0, 1.0, (n, 1 + 8 + 28)), 2)
    if scan == "pruned":
        gpu.table_set_scan(t, gpu.SCAN_PRUNED)
    out = []
    for step in (gpu.chains_step, gpu.chains_step_profiled):
        net = gpu.mlp_create(n, synth.mlp_init_weights(n, 8, 128, 3), hidden=128, d=8, batch_cap=C, lr=1e-2)
        ch = gpu.chains_create(t, C, 5)
        gpu.chains_set_proposal(ch, net, gpu.PROPOSAL_TRAIN)
        step(ch, 5)
        gpu.mlp_adam_step(net)
        step(ch, 1)
        step(ch, 4)
        out.append(_weights(gpu, net))
    for x in TENSORS:
        assert np.array_equal(out[0][x], out[1][x]), x


def test_corrections_follow_the_step_count(gpu):
    """One gradient, many Adam steps: b3 against the recurrence in FP64.  The gradient is the
    same every step, so moments and corrections cancel and a step is lr g / (|g| + eps); FP32
    rounding leaves a few 2^-24 of lr a step and of the weight."""
    n, B, lr, steps = 8, 30, 1e-2, 25
    net = gpu.mlp_create(n, synth.mlp_init_weights(n, 8, 128, 3), hidden=128, d=8, batch_cap=B, lr=lr)
    rng = np.random.default_rng(4)
    gpu.mlp_loss_grad(net, synth.random_orders(n, B, 1), rng.integers(0, 28, B).astype(np.uint32),
                      rng.random(B).astype(np.float32))
    g = gpu.mlp_read(net, "b3", grad=True).astype(np.float64)
    w = gpu.mlp_read(net, "b3").astype(np.float64)
    m = v = np.zeros_like(w)
    b1, b2, eps = float(np.float32(0.9)), float(np.float32(0.999)), float(np.float32(1e-8))
    for s in range(1, steps + 1):
        gpu.mlp_adam_step(net)
        m = b1 * m + (1 - b1) * g
        v = b2 * v + (1 - b2) * g * g
        w = w - float(np.float32(lr)) * (m / (1 - b1 ** s)) / (np.sqrt(v / (1 - b2 ** s)) + eps)
    # 1 - b2 and 1 - b2^s in FP32 carry 2^-24 of 1 into numbers from 0.001 on: 6e-5, its square root 3e-5
    assert np.abs(gpu.mlp_read(net, "b3") - w).max() <= steps * lr * 1e-4 + 1e-6
