"""The sum-based order score where its window of counted entries can go wrong: tables whose
every entry counts, tables where only the best does, ties, -inf entries, window ends at
chunk edges, batches around the block's eight orders and the partials' 256, k above 4 (no
bit-sliced scan for the best entries) and a pruned table.

Against a host log-sum-exp in FP64; the bar is 1e-12 relative per node term and order, as for
the oracle comparison (the same FP64 terms in another order; what lies outside the window
is below 2^-60 of a sum)."""
import itertools

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _ref(sc, masks, order):
    out, pred = np.empty(len(order)), 0
    for v in order:
        v = int(v)
        pc = (pred & ((1 << v) - 1)) | (pred >> (v + 1) << v)
        x = sc[v][(masks & ~pc) == 0]
        m = x.max()
        out[v] = m if np.isneginf(m) else m + np.log10(np.sum(10.0 ** (x - m)))
        pred |= 1 << v
    return out


@pytest.mark.parametrize("kind", ["flat", "steep", "ties", "inf", "decades"])
@pytest.mark.parametrize("n,k,B,pruned", [(6, 2, 1, False), (14, 4, 9, False), (19, 4, 8, True), (16, 5, 17, False),
                                          (22, 4, 300, False)])
def test_sum_window(gpu, n, k, B, pruned, kind):
    rng = np.random.default_rng(n + len(kind))
    S = oracle.num_sets(n - 1, k)
    sc = {"flat": lambda: -3.0 - rng.random((n, S)) * 1e-3,
          "steep": lambda: -1e5 * rng.random((n, S)),
          "ties": lambda: rng.choice([-40.0, -20.0, -8.0], (n, S)),
          "inf": lambda: np.where(rng.random((n, S)) < 0.3, -np.inf, -30.0 * rng.random((n, S))),
          "decades": lambda: -60.0 * rng.random((n, S)) - 500.0}[kind]()
    masks = np.array([sum(1 << c for c in cs) for j in range(k + 1)
                      for cs in sorted(itertools.combinations(range(n - 1), j), key=lambda c: c[::-1])], np.int64)
    t = gpu.table_from_scores(sc, k)
    if pruned:
        gpu.table_set_scan(t, gpu.SCAN_PRUNED)
    orders = synth.random_orders(n, B, 5)
    tot, node = gpu.score_orders_sum(t, orders)
    for b in range(0, B, max(1, B // 20)):
        ref = _ref(sc, masks, orders[b])
        np.testing.assert_allclose(node[b], ref, rtol=1e-12, atol=1e-12)
        np.testing.assert_allclose(tot[b], ref.sum(), rtol=1e-12)
    tot2, node2 = gpu.score_orders_sum(t, orders)
    assert np.array_equal(node, node2) and np.array_equal(tot, tot2)
