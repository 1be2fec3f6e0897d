"""The ranking of a table's entries (sorted positions, their inverse, the sorted parent sets)
on score distributions and sizes where the bucket sort can go wrong: ties of every extent,
scores packed into one narrow range beside far outliers, -inf, already sorted input, one
bucket (a node's entries sorted by one block) and many, and the radix sort above 2 M sets.

The ranking is not an output of its own; every scan mode reads it.  Each mode's chosen
parent sets and scores must equal a brute-force maximum (ties to the lowest rank) exactly."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _scores(kind, n, S, rng):
    x = rng.normal(-500.0, 40.0, (n, S))
    if kind == "equal":
        x[:] = -7.25
    elif kind == "few":
        x = rng.choice([-3.0, -2.0, -1.0, 0.0], (n, S))
    elif kind == "outlier":
        x = -1.0 - rng.random((n, S)) * 1e-9
        x[:, S // 2] = -1e300
        x[:, S // 3] = 1e300
        x[:, S // 5] = -np.inf
    elif kind == "ascending":
        x = np.sort(x, axis=1)
    elif kind == "descending":
        x = -np.sort(-x, axis=1)
    elif kind == "cluster":
        x = np.where(rng.random((n, S)) < 0.9, -100.0 + rng.integers(0, 3, (n, S)) * 2.0 ** -40, x)
    return x


@pytest.mark.parametrize("kind", ["normal", "equal", "few", "outlier", "ascending", "descending", "cluster"])
@pytest.mark.parametrize("n,k", [(6, 2), (17, 4), (19, 4), (20, 4), (30, 4)])     # 16 .. 27,841 sets a node
def test_ranking(gpu, n, k, kind):
    rng = np.random.default_rng(7 * n + len(kind))
    S = oracle.num_sets(n - 1, k)
    sc = _scores(kind, n, S, rng)
    orders = synth.random_orders(n, 40, n)
    ref = [oracle.order_score(sc, k, o) for o in orders]
    t = gpu.table_from_scores(sc, k)
    for mode in (gpu.SCAN_FULL, gpu.SCAN_SLICED, gpu.SCAN_SORTED, gpu.SCAN_PRUNED):
        gpu.table_set_scan(t, mode)
        br, s = gpu.score_orders(t, orders)
        for b in range(len(orders)):
            assert np.array_equal(br[b], ref[b][1]) and s[b] == ref[b][0], (mode, b)


def test_ranking_above_two_million_sets(gpu):
    import torch
    n, k = 23, 11
    S = oracle.num_sets(n - 1, k)
    assert S > 2 * 1024 * 1024
    g = torch.Generator(device="cuda").manual_seed(5)
    sc = torch.randint(-1000000, 0, (n, S), generator=g, device="cuda", dtype=torch.int64).double()     # many ties
    t = gpu.table_from_scores(sc, k)
    assert gpu.table_info(t)["sets_per_node"] == S
    masks = torch.cat([_colex(n - 1, j) for j in range(k + 1)])
    orders = synth.random_orders(n, 12, 3)
    br, s = gpu.score_orders(t, orders)
    for b, o in enumerate(orders):
        pred, tot = 0, 0.0
        best = {}
        for v in o:
            v = int(v)
            pc = (pred & ((1 << v) - 1)) | (pred >> (v + 1) << v)
            x = torch.where((masks & ~pc) == 0, sc[v], torch.full((), -np.inf, dtype=torch.float64, device="cuda"))
            m = x.max()
            best[v] = (int((x == m).nonzero()[0]), float(m))
            pred |= 1 << v
        for v in range(n):
            assert br[b][v] == best[v][0]
            tot += best[v][1]
        assert s[b] == tot


def _colex(N, j):
    """Masks of the j-subsets of range(N) in colex order = ascending mask order."""
    import torch
    m = torch.arange(1 << N, device="cuda", dtype=torch.int64)
    c = torch.zeros_like(m)
    for t in range(N):
        c += (m >> t) & 1
    return m[c == j]
