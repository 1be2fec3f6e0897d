"""Ranking where a bucket's scores tie or crowd and its block sorts it by a network: bucket sizes
of one entry, at and around powers of two, a whole block's capacity (4,096 sets a node) and
several buckets, ties that reach across buckets, and two crowded values inside a spread.  The
chosen parent sets equal a brute-force maximum (ties to the lowest rank) exactly.

And its cost: by the network's length (66 steps for 2,048 entries, of a pair each) equal
scores rank within four times the time of scores that are all different."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _scores(kind, n, S, rng):
    if kind == "equal":
        return np.full((n, S), -3.5)
    if kind == "two":
        return rng.choice([-2.0, -1.0], (n, S))
    if kind == "falling":                             # runs of equal scores, the best last
        return np.floor(np.arange(n * S).reshape(n, S) % S / 300.0) - 1000.0
    x = rng.normal(-50.0, 9.0, (n, S))                # crowded values beside different ones
    return np.where(rng.random((n, S)) < 0.8, rng.choice([-40.0, -40.0 - 2.0 ** -47], (n, S)), x)


@pytest.mark.parametrize("kind", ["equal", "two", "falling", "crowd"])
@pytest.mark.parametrize("n,k", [(4, 0), (2, 1), (9, 7), (9, 8), (12, 10), (12, 11), (13, 11), (13, 12), (14, 13),
                                 (20, 4), (27, 4), (17, 8)])     # 1, 2, 255, 256, ... 4,095, 4,096, 8,192 sets ...
def test_ties(gpu, n, k, kind):
    rng = np.random.default_rng(n * 100 + k)
    S = oracle.num_sets(n - 1, k)
    sc = _scores(kind, n, S, rng)
    t = gpu.table_from_scores(sc, k)
    orders = synth.random_orders(n, 24, n + k)
    ref = [oracle.order_score(sc, k, o) for o in orders]
    for mode in [gpu.SCAN_FULL] + ([gpu.SCAN_PRUNED] if k <= 7 else []) + ([gpu.SCAN_SORTED] if k <= 4 else []):
        gpu.table_set_scan(t, mode)
        br, s = gpu.score_orders(t, orders)
        for b in range(len(orders)):
            assert np.array_equal(br[b], ref[b][1]) and s[b] == ref[b][0], (mode, b)


@pytest.mark.parametrize("n,k", [(60, 4), (40, 5)])              # 489,406 and 667,966 sets a node
def test_equal_scores_are_not_slow(gpu, n, k):
    import torch
    S = oracle.num_sets(n - 1, k)
    g = torch.Generator(device="cuda").manual_seed(1)
    ms = []
    for sc in (torch.rand((n, S), generator=g, device="cuda", dtype=torch.float64),
               torch.full((n, S), -1.0, device="cuda", dtype=torch.float64)):
        t = []
        for _ in range(7):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            tab = gpu.table_from_scores(sc, k)
            e[1].record()
            e[1].synchronize()
            tab.free()
            t.append(e[0].elapsed_time(e[1]))
        ms.append(sorted(t)[3])
    assert ms[1] < 4 * ms[0], ms
