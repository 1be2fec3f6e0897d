"""Learned steps of more chains than fit on the GPU at once, stepped in groups: a chain's
trajectory depends on its number and the seed alone, so the first chains of a large set equal
those of a small one bit for bit, whatever the launch, every order stays a permutation, and the
set's step counter, trace and records are those of one group."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,H,C,launch", [(60, 128, 2048, "AUTO"), (47, 128, 1025, "AUTO"), (60, 256, 700, "AUTO"),
                                          (60, 256, 700, "GRAPH"), (60, 640, 385, "AUTO")])
def test_first_chains_of_a_large_set(gpu, n, H, C, launch):
    rng = np.random.default_rng(C)
    few, calls = 130, (60, 1, 39)
    t = gpu.table_from_scores(rng.normal(-500.0, 4.0, (n, 1 + (n - 1) + (n - 1) * (n - 2) // 2)), 2)
    gpu.table_set_scan(t, gpu.SCAN_PRUNED)
    w = synth.mlp_init_weights(n, 8, H, 3)
    what = ("orders", "scores", "ranks", "best_scores", "best_orders", "best_ranks", "accepts", "edge_counts", "logits",
            "trace_score", "trace_accept", "record")
    out = []
    for chains in (few, C):
        net = gpu.mlp_create(n, w, hidden=H, d=8, batch_cap=chains)
        ch = gpu.chains_create(t, chains, 9, burn_in=5, trace_cap=80, record_every=10, record_cap=16)
        gpu.chains_set_proposal(ch, net, gpu.PROPOSAL_LEARNED, eps_mix=0.1)
        gpu.chains_set_learned_launch(ch, getattr(gpu, "LEARNED_LAUNCH_" + launch))
        for steps in calls:
            gpu.chains_step(ch, steps)
        out.append({x: gpu.chains_read(ch, x) for x in what})
        assert (np.sort(out[-1]["orders"], axis=1) == np.arange(n)).all()
        assert gpu.chains_read(ch, "steps")[0] == sum(calls)
    for x in what:
        assert np.array_equal(out[0][x], out[1][x][:few]), x
    assert out[1]["accepts"].min() >= 0 and out[1]["accepts"].sum() > C
