"""The persistent learned step hands its phases on per 128 chains: chain counts around whole
tiles and blocks of four, with an output layer wide enough (47 nodes: 34 tiles) that chain
blocks sit with output tiles of the same chains, and one that is not.  Bit for bit what the
three kernels per step give."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,H,C", [(47, 128, 1), (47, 128, 127), (47, 128, 128), (47, 128, 129), (48, 128, 301), (30, 128, 259)])
def test_phases_equal_graph_launch(gpu, n, H, C):
    rng = np.random.default_rng(n + C)
    k, steps = 2, 300
    S = 1 + (n - 1) + (n - 1) * (n - 2) // 2
    t = gpu.table_from_scores(rng.normal(-500.0, 3.0, (n, S)), k)
    gpu.table_set_scan(t, gpu.SCAN_PRUNED)
    w = synth.mlp_init_weights(n, 8, H, 3)
    out = []
    for mode in (gpu.LEARNED_LAUNCH_GRAPH, gpu.LEARNED_LAUNCH_AUTO):
        net = gpu.mlp_create(n, w, hidden=H, d=8, batch_cap=C)
        ch = gpu.chains_create(t, C, 5, burn_in=10, trace_cap=steps)
        gpu.chains_set_learned_launch(ch, mode)
        gpu.chains_set_proposal(ch, net, gpu.PROPOSAL_LEARNED, eps_mix=0.2)
        gpu.chains_step(ch, steps)
        out.append({what: gpu.chains_read(ch, what) for what in
                    ("trace_score", "trace_accept", "orders", "scores", "ranks", "best_scores", "best_orders",
                     "accepts", "edge_counts", "steps", "items", "logits")})
    for what in out[0]:
        assert np.array_equal(out[0][what], out[1][what]), what
