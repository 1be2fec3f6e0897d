"""The joint counts of the largest sets on the tensor cores where their tiles can go wrong:
row counts around a stage (128) and a word, every mix of arities (pairs of 4 to 16 and low
sets of 4 to 64 states, tiles that end inside a pair block or a set), both set sizes
(k = 3: pairs by pairs, k = 4: pairs by triples, and pairs by pairs once more for the parent
sets of four nodes, with one to three variants of the configuration sums), one lgamma table
for all (K2, BDeu with one arity), rows up to where the tables fill the shared memory, and
the networks around the size from which they are used.

Every entry against the oracle: 1e-12 relative, as for every table entry (counts and
fixed-point sums are exact; one rounding)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k,m,arities,kind", [
    (26, 4, 64, (2, 3, 4), 0), (27, 4, 127, (3,), 1), (26, 4, 128, (2,), 1), (27, 4, 129, (4,), 0),
    (26, 4, 300, (3,), 0), (28, 4, 1000, (2, 4), 0), (37, 3, 65, (2, 3, 4), 0), (38, 3, 500, (4,), 1),
    (37, 3, 255, (2,), 0), (29, 4, 1574, (2, 3, 4), 0), (28, 4, 2099, (2, 3), 0), (27, 4, 3149, (3,), 1),
    (27, 4, 1575, (2, 3, 4), 0), (37, 3, 6299, (2, 3), 0), (37, 3, 6300, (3,), 0),
    (36, 4, 300, (2, 3, 4), 0), (36, 4, 257, (2, 4), 0), (37, 4, 200, (3,), 1), (36, 4, 64, (2,), 0),
    (36, 4, 1574, (2, 3, 4), 0), (39, 3, 3599, (3, 4), 0), (37, 3, 3600, (2, 3), 0), (25, 4, 500, (3,), 0), (36, 3, 500, (2, 3), 0)])
def test_tensor_core_counts(gpu, n, k, m, arities, kind):
    rng = np.random.default_rng(n * 1000 + m)
    ar = rng.choice(arities, n).astype(np.uint8)
    # skewed columns, some constant: counts from 0 to m
    x = np.stack([np.minimum(rng.geometric(rng.uniform(0.3, 1.0), m) - 1, a - 1) for a in ar], 1).astype(np.uint8)
    R = rng.random((n, n))
    t = gpu.build_scores(x, ar, k, R=R, score_kind=kind, ess=2.0)
    ref = oracle.build_table(x, ar, k, kind, 2.0, 0.0, R, threads=None)
    np.testing.assert_allclose(gpu.table_scores(t), ref, rtol=1e-12, atol=1e-12)
