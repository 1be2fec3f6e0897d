"""The table build through joint count tables against the oracle, where its splits can go
wrong: joint sets over all 64 nodes (masks with every bit), sets that hold every node,
work units that end inside a run of sets, and the launch shapes with fewer warps a block
and without the row bases (tens of thousands of rows).

Bar: 1e-12 relative, as for every table entry (exact fixed-point sums of the FP64 lgamma
terms, one rounding, against the oracle's FP64 sums)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _data(n, m, seed, arities=(2, 3, 4)):
    rng = np.random.default_rng(seed)
    ar = rng.choice(arities, n).astype(np.uint8)
    x = np.stack([np.minimum(rng.geometric(0.5, m) - 1, a - 1) for a in ar], 1).astype(np.uint8).reshape(m, n)
    return x, ar


@pytest.mark.parametrize("n,k,m", [(64, 2, 70), (64, 1, 33), (63, 2, 5), (2, 1, 40), (5, 4, 129), (9, 5, 64),
                                   (7, 3, 30000), (4, 2, 70000)])
@pytest.mark.parametrize("kind", [0, 1])
def test_joint_build(gpu, n, k, m, kind):
    data, ar = _data(n, m, 100 * n + k, (2, 3) if k >= 5 else (2, 3, 4))
    R = np.random.default_rng(n).random((n, n))
    t = gpu.build_scores(data, ar, k, R=R, score_kind=kind, ess=3.0, log10_gamma=-0.25)
    ref = oracle.build_table(data, ar, k, kind, 3.0, -0.25, R, threads=None)
    np.testing.assert_allclose(gpu.table_scores(t), ref, rtol=1e-12, atol=1e-12)


def test_one_arity_present(gpu):
    # K2 keeps one configuration sum per child arity present; here the only one is 4
    data, _ = _data(6, 200, 9)
    ar = np.full(6, 4, np.uint8)
    t = gpu.build_scores(data, ar, 3)
    np.testing.assert_allclose(gpu.table_scores(t), oracle.build_table(data, ar, 3), rtol=1e-12, atol=1e-12)
