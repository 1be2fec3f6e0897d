"""The survivors of dominance pruning, counted entry by entry on the host: size classes of
every kind the pruning has a kernel for (k = 0 .. 7), chunk edges of the compaction, many
survivors and few.  Counts are whole numbers and must be equal."""
import itertools

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _survivors(sc, N, k):
    """Per node, the entries that no proper subset of their set matches or beats."""
    sets = [c for j in range(k + 1) for c in sorted(itertools.combinations(range(N), j), key=lambda c: c[::-1])]
    rank = {c: r for r, c in enumerate(sets)}
    out = []
    for row in sc:
        best, alive = {}, 0
        for c in sets:
            sub = max((best[c[:t] + c[t + 1:]] for t in range(len(c))), default=-np.inf)
            alive += len(c) == 0 or row[rank[c]] > sub
            best[c] = max(sub, row[rank[c]])
        out.append(alive)
    return out


@pytest.mark.parametrize("n,k", [(2, 1), (5, 0), (9, 1), (12, 3), (18, 4), (12, 5), (10, 6), (10, 7)])
@pytest.mark.parametrize("kind", ["random", "ties", "rising"])
def test_survivor_counts(gpu, n, k, kind):
    rng = np.random.default_rng(n * 10 + k)
    S = oracle.num_sets(n - 1, k)
    sc = rng.normal(-50, 10, (n, S)) if kind == "random" else rng.integers(-4, 0, (n, S)).astype(float)
    if kind == "rising":
        sc = np.sort(rng.normal(-50, 10, (n, S)), axis=1)       # every entry survives
    t = gpu.table_from_scores(sc, k)
    gpu.table_set_scan(t, gpu.SCAN_PRUNED)
    assert list(gpu.table_pruned(t)) == _survivors(sc, n - 1, k)
