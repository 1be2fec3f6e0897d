"""The histogram counts on either side of the rule that keeps the rows' offsets in shared
memory: rows around 2,500 with sets enough for it and with too few, k = 5 around the rows
with which two blocks still fit an SM, and the rows between what the tensor cores take
(6,300) and what a row list can name (16,384), and around both.  Every entry against the
oracle: 1e-12 relative, as for every table entry.

And their cost: more rows must not take over-proportionally long.  The work of a set grows
with its rows, so 16,000 rows may take no more than 16 times what 1,000 take (and fixed work
makes it less)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _data(n, m, arities, seed):
    rng = np.random.default_rng(seed)
    ar = rng.choice(arities, n).astype(np.uint8)
    x = np.stack([np.minimum(rng.geometric(rng.uniform(0.3, 0.9), m) - 1, a - 1) for a in ar], 1).astype(np.uint8)
    return x, ar


@pytest.mark.parametrize("n,k,m,arities,kind", [
    (30, 4, 2500, (2, 3, 4), 1), (30, 4, 2501, (2, 3, 4), 1), (30, 4, 1000, (2, 3), 1), (27, 4, 777, (2, 3, 4), 1),
    (26, 4, 100, (2, 3, 4), 1), (28, 4, 333, (4,), 0),
    (14, 5, 3000, (2, 3), 1), (12, 5, 6784, (2,), 0), (12, 5, 6785, (2,), 0), (12, 5, 6900, (2,), 1), (9, 5, 1, (2, 3), 0),
    (10, 4, 6299, (3,), 0), (10, 4, 6301, (2, 3, 4), 0), (9, 3, 8000, (2, 3, 4), 1), (11, 3, 12001, (2, 3, 4), 0),
    (8, 4, 16383, (4,), 0), (8, 4, 16384, (2, 3, 4), 1), (8, 4, 16385, (2, 3, 4), 0), (6, 5, 16384, (2, 3), 1)])
def test_rows_and_sets(gpu, n, k, m, arities, kind):
    x, ar = _data(n, m, arities, 1000 * n + m)
    t = gpu.build_scores(x, ar, k, score_kind=kind, ess=2.0)
    ref = oracle.build_table(x, ar, k, kind, 2.0, 0.0, None, threads=None)
    np.testing.assert_allclose(gpu.table_scores(t), ref, rtol=1e-12, atol=1e-12)


@pytest.mark.parametrize("n,k,arities,kind", [(30, 3, (3,), 0), (37, 4, (2, 3, 4), 1), (60, 2, (2, 3, 4), 0), (20, 4, (2, 3, 4), 1)])
def test_many_rows_are_not_slow(gpu, n, k, arities, kind):
    ms = []
    for m in (1000, 16000):
        x, ar = _data(n, m, arities, n)
        ms.append(sorted(gpu.build_scores_profiled(x, ar, k, score_kind=kind)[1] for _ in range(6))[2])
    assert ms[1] < 16 * ms[0], ms
