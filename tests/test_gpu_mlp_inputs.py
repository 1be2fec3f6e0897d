"""Orders and swap pairs that do not exist are refused (BN_EINVAL) by the proposal network's
forward and backward passes, on host and device arrays, and leave nothing behind: the next
valid call gives the same bits as on a network that never saw them."""
import ctypes as C

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", ["node_n", "node_255", "pair_P", "pair_huge"])
@pytest.mark.parametrize("row", [0, 36])
def test_inputs_that_do_not_exist(gpu, bad, row):
    n, B, H = 11, 37, 128
    P = n * (n - 1) // 2
    rng = np.random.default_rng(1)
    w = synth.mlp_init_weights(n, 8, H, 3)
    nets = [gpu.mlp_create(n, w, hidden=H, d=8, batch_cap=B) for _ in range(2)]
    o, p = synth.random_orders(n, B, 4), rng.integers(0, P, B).astype(np.uint32)
    a = rng.random(B).astype(np.float32)
    o2, p2 = o.copy(), p.copy()
    if bad.startswith("node"):
        o2[row, n - 1] = n if bad == "node_n" else 255
        with pytest.raises(gpu.BNError) as e:
            gpu.mlp_forward(nets[0], o2)
        assert e.value.code == gpu.EINVAL
    else:
        p2[row] = P if bad == "pair_P" else 0xffffffff
    with pytest.raises(gpu.BNError) as e:
        gpu.mlp_loss_grad(nets[0], o2, p2, a)
    assert e.value.code == gpu.EINVAL
    import torch
    d = [torch.from_numpy(x).cuda() for x in (o2, p2.view(np.int32), a)]
    loss = torch.zeros(1, device="cuda")
    rc = gpu.lib().bn_mlp_loss_grad(nets[0].handle, *[C.c_void_p(x.data_ptr()) for x in d], B, C.c_void_p(loss.data_ptr()),
                                    gpu.MEM_DEVICE, None)
    assert rc == gpu.EINVAL
    for net in nets:
        for _ in range(2):
            gpu.mlp_loss_grad(net, o, p, a)
            gpu.mlp_adam_step(net)
    assert np.array_equal(gpu.mlp_forward(nets[0], o), gpu.mlp_forward(nets[1], o))
    for x in ("E", "W1", "b1", "W2", "b2", "W3", "b3"):
        assert np.array_equal(gpu.mlp_read(nets[0], x), gpu.mlp_read(nets[1], x)), x
        assert np.array_equal(gpu.mlp_read(nets[0], x, grad=True), gpu.mlp_read(nets[1], x, grad=True)), x
