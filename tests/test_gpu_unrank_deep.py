"""BN_SCAN_UNRANK on tables made from scores whose parent sets exceed the builder's twelve
nodes: the binomials in shared memory follow the table's k.  Bit for bit the oracle."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k", [(14, 12), (14, 13), (16, 14), (17, 16)])
def test_unranked_sets_above_twelve_parents(gpu, n, k):
    rng = np.random.default_rng(n * k)
    sc = rng.normal(-100.0, 5.0, (n, oracle.num_sets(n - 1, k)))
    t = gpu.table_from_scores(sc, k)
    gpu.table_set_scan(t, gpu.SCAN_UNRANK)
    orders = synth.random_orders(n, 9, n)
    best, score = gpu.score_orders(t, orders)
    for b in range(len(orders)):
        s, r = oracle.order_score(sc, k, orders[b])
        assert np.array_equal(best[b], r) and score[b] == s, b
