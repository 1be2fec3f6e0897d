"""Two chain sets with networks of different width used in turn: the persistent launch of the
wider one keeps its shared memory after the narrower one has been set up.  Each set's states
equal those of a set stepped alone by the three kernels per step, bit for bit, and the
persistent launch is the one that ran."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _set(gpu, t, n, H, C, mode):
    net = gpu.mlp_create(n, synth.mlp_init_weights(n, 8, H, 5), hidden=H, d=8, batch_cap=C)
    ch = gpu.chains_create(t, C, 3)
    gpu.chains_set_learned_launch(ch, mode)
    gpu.chains_set_proposal(ch, net, gpu.PROPOSAL_LEARNED, eps_mix=0.2)
    return net, ch


def test_wider_network_steps_again_after_a_narrower_one(gpu):
    n, C, steps = 20, 40, 60
    rng = np.random.default_rng(0)
    t = gpu.table_from_scores(rng.normal(-300.0, 2.0, (n, 1 + 19 + 19 * 9)), 2)
    gpu.table_set_scan(t, gpu.SCAN_PRUNED)
    what = ("orders", "scores", "ranks", "accepts", "edge_counts", "logits")
    ref = {}
    for H in (512, 128):
        net, ch = _set(gpu, t, n, H, C, gpu.LEARNED_LAUNCH_GRAPH)
        gpu.chains_step(ch, 2 * steps)
        ref[H] = {w: gpu.chains_read(ch, w) for w in what}
    wide = _set(gpu, t, n, 512, C, gpu.LEARNED_LAUNCH_AUTO)
    narrow = _set(gpu, t, n, 128, C, gpu.LEARNED_LAUNCH_AUTO)
    for _ in range(2):
        for _, ch in (wide, narrow):
            before = gpu.kernel_launches()
            gpu.chains_step(ch, steps)
            assert gpu.kernel_launches() - before < steps
    for H, (_, ch) in ((512, wide), (128, narrow)):
        for w in what:
            assert np.array_equal(gpu.chains_read(ch, w), ref[H][w]), (H, w)
