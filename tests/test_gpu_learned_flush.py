"""Edge counts of learned steps that end a call on an accepted swap: the accept starts new
dwells from the lanes of its positions, and the flush credits every node's dwell from the
lane of its id.  With one step a call, every accept meets a flush; the counts must equal the
number of recorded steps that hold each edge, exactly."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,C,calls", [(9, 5, [1] * 60), (40, 33, [1] * 40 + [2, 1, 3]), (64, 7, [1] * 30)])
def test_edge_counts_of_single_step_calls(gpu, n, C, calls):
    rng = np.random.default_rng(n)
    S = 1 + (n - 1) + (n - 1) * (n - 2) // 2
    t = gpu.table_from_scores(rng.normal(-5.0, 0.2, (n, S)), 2)         # most swaps are accepted
    gpu.table_set_scan(t, gpu.SCAN_PRUNED)
    out = []
    for mode in (gpu.LEARNED_LAUNCH_GRAPH, gpu.LEARNED_LAUNCH_AUTO):
        net = gpu.mlp_create(n, synth.mlp_init_weights(n, 8, 128, 3), hidden=128, d=8, batch_cap=C)
        ch = gpu.chains_create(t, C, 11, record_every=1, record_cap=sum(calls))
        gpu.chains_set_learned_launch(ch, mode)
        gpu.chains_set_proposal(ch, net, gpu.PROPOSAL_LEARNED, eps_mix=0.3)
        for steps in calls:
            gpu.chains_step(ch, steps)
        assert gpu.chains_read(ch, "accepts").sum() > sum(calls)
        assert gpu.chains_read(ch, "record_len")[0] == sum(calls)
        bits = gpu.chains_read(ch, "record")
        held = np.unpackbits(bits.view(np.uint8).reshape(C, n, n, -1), axis=3).sum(3)
        counts = gpu.chains_read(ch, "edge_counts")
        assert np.array_equal(counts, held)
        out.append(counts)
    assert np.array_equal(out[0], out[1])
