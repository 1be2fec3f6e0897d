"""Which kernel scans a batch must not show: sizes on both sides of every line that chooses
one (sets per node, orders, (node, order) items, slices per SM), in the default scan mode,
against the pruned scan, itself against the oracle elsewhere, and the oracle on a sample.
Chosen parent sets and FP64 scores are equal bit for bit."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k", [(6, 4), (13, 4), (19, 4), (20, 4), (22, 4), (23, 4), (33, 3), (15, 5), (18, 6)])
def test_default_scan_routes(gpu, n, k):
    rng = np.random.default_rng(n)
    S = oracle.num_sets(n - 1, k)
    sc = np.round(rng.normal(-200.0, 15.0, (n, S)), 1)              # with ties
    t = gpu.table_from_scores(sc, k)
    p = gpu.table_from_scores(sc, k)
    gpu.table_set_scan(p, gpu.SCAN_PRUNED)
    for B in (1, 3, 4, 15, 16, 31, 33, 64, 65, 127, 129, 256, 257, 600):
        orders = synth.random_orders(n, B, 100 + B)
        br, s = gpu.score_orders(t, orders)
        br2, s2 = gpu.score_orders(p, orders)
        assert np.array_equal(br, br2) and np.array_equal(s, s2), B
        b = B - 1
        ref = oracle.order_score(sc, k, orders[b])
        assert s[b] == ref[0] and np.array_equal(br[b], ref[1])


@pytest.mark.parametrize("n", [20, 24, 30])                          # below and above the list rule
@pytest.mark.parametrize("chains", [1, 5, 40, 300])
def test_default_scan_sampler(gpu, n, chains):
    rng = np.random.default_rng(n)
    sc = rng.normal(-200.0, 3.0, (n, oracle.num_sets(n - 1, 4)))
    t = gpu.table_from_scores(sc, 4)
    out = []
    for mode in (gpu.SCAN_FULL, gpu.SCAN_PRUNED):
        gpu.table_set_scan(t, mode)
        c = gpu.chains_create(t, chains, seed=3, burn_in=5)
        gpu.chains_step(c, 40)
        out.append([gpu.chains_read(c, w) for w in ("orders", "scores", "best_ranks", "edge_counts", "accepts")])
    assert all(np.array_equal(a, b) for a, b in zip(*out))
