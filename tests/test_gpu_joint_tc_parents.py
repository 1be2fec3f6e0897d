"""Parent sets of four nodes counted on the tensor cores with every number of variants of the
configuration sums (K2 with one, two and three arities present, BDeu), at rows around a stage
and up to where four lgamma tables fill the shared memory, on either side of the line from
which they are used (C(37, 4) = 66,045 sets; C(36, 4) = 58,905 are too few).

That they ran is checked by the launches: each size of set on the tensor cores takes two
(states, counts) over the same build without (63 rows; one more there where the rows' offsets
are kept).  Every entry against the oracle: 1e-12 relative, as for every table entry."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _build(gpu, x, ar, k, kind):
    before = gpu.kernel_launches()
    t = gpu.build_scores(x, ar, k, score_kind=kind, ess=2.0)
    return t, gpu.kernel_launches() - before


@pytest.mark.parametrize("n,m,arities,kind,sizes", [
    (37, 300, (2, 3, 4), 0, 2), (37, 129, (2, 4), 0, 2), (38, 64, (2, 3), 0, 2), (37, 127, (4, 3), 0, 2),
    (37, 1574, (2, 3, 4), 0, 2), (37, 1575, (2, 3, 4), 0, 1), (37, 257, (2,), 0, 2), (38, 200, (3,), 1, 2),
    (36, 130, (2, 3, 4), 0, 1), (37, 130, (2, 3, 4), 1, 0)])
def test_variants(gpu, n, m, arities, kind, sizes):
    k = 4
    rng = np.random.default_rng(n * 1000 + m)
    ar = rng.choice(arities, n).astype(np.uint8)
    assert set(ar) == set(arities)
    x = np.stack([np.minimum(rng.geometric(rng.uniform(0.3, 1.0), m) - 1, a - 1) for a in ar], 1).astype(np.uint8)
    _, without = _build(gpu, x[:63], ar, k, kind)
    t, launches = _build(gpu, x, ar, k, kind)
    assert (launches - (without & ~1)) // 2 == sizes, (launches, without)
    ref = oracle.build_table(x, ar, k, kind, 2.0, 0.0, None, threads=None)
    np.testing.assert_allclose(gpu.table_scores(t), ref, rtol=1e-12, atol=1e-12)
