"""The sizes at which the persistent learned step is compared with the graph (47 nodes: 1,081
swap pairs, 36 output tiles) do take the persistent launch in the automatic mode: a call of
many steps launches far fewer kernels than steps, the graph three a step."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,H,C", [(47, 128, 1), (47, 128, 129), (48, 128, 301), (30, 128, 259), (60, 512, 256)])
def test_auto_is_persistent(gpu, n, H, C):
    rng = np.random.default_rng(n + C)
    steps = 300
    t = gpu.table_from_scores(rng.normal(-500.0, 3.0, (n, 1 + (n - 1) + (n - 1) * (n - 2) // 2)), 2)
    gpu.table_set_scan(t, gpu.SCAN_PRUNED)
    for mode, low, high in ((gpu.LEARNED_LAUNCH_AUTO, 1, steps // 4), (gpu.LEARNED_LAUNCH_GRAPH, 3 * steps, 4 * steps)):
        net = gpu.mlp_create(n, synth.mlp_init_weights(n, 8, H, 3), hidden=H, d=8, batch_cap=C)
        ch = gpu.chains_create(t, C, 5)
        gpu.chains_set_learned_launch(ch, mode)
        gpu.chains_set_proposal(ch, net, gpu.PROPOSAL_LEARNED, eps_mix=0.2)
        before = gpu.kernel_launches()
        gpu.chains_step(ch, steps)
        assert low <= gpu.kernel_launches() - before <= high, mode
