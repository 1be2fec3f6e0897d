"""Buckets that outgrow a block's shared memory (4,096 entries).  The splitters come from a
fixed pseudo-random sample of positions; scores that put every sampled entry above all others
leave the rest in one bucket.  The sampling is restated here, the bucket's size checked, and
the chosen parent sets compared with a brute-force maximum exactly."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
CAP = 4096


def _sampled(S):
    """Positions of the sample and the splitters' places in it, as the ranking takes them."""
    NB = min(1024, -(-S // 1024))
    M = 32
    while M < 8 * NB and M < 8192:
        M *= 2
    j = np.arange(M, dtype=np.uint64)
    lo, hi = S * j // M, S * (j + 1) // M
    u32 = np.uint64(0xffffffff)
    h = j * np.uint64(0x9E3779B9) & u32
    h ^= h >> np.uint64(15)
    h = h * np.uint64(0x85EBCA6B) & u32
    h ^= h >> np.uint64(13)
    return (lo + h % (hi - lo)).astype(np.int64), [M * (b + 1) // NB for b in range(NB - 1)]


@pytest.mark.parametrize("n,k", [(20, 4), (24, 4)])              # 5,036 and 10,903 sets a node
@pytest.mark.parametrize("kind", ["distinct", "ties"])
def test_oversized_bucket(gpu, n, k, kind):
    rng = np.random.default_rng(n)
    S = oracle.num_sets(n - 1, k)
    pos, cuts = _sampled(S)
    sc = rng.normal(-900.0, 5.0, (n, S)) if kind == "distinct" else rng.choice([-900.0, -901.0, -905.5], (n, S))
    top = rng.normal(-100.0, 1.0, (n, len(pos)))
    sc[:, pos] = top if kind == "distinct" else np.round(top)
    for i in range(n):
        order = np.lexsort((pos, -sc[i, pos]))
        last = sc[i, pos[order[cuts[-1]]]]                       # the last splitter
        assert (sc[i] < last).sum() > CAP
    t = gpu.table_from_scores(sc, k)
    orders = synth.random_orders(n, 40, 2)
    ref = [oracle.order_score(sc, k, o) for o in orders]
    for mode in (gpu.SCAN_FULL, gpu.SCAN_SLICED, gpu.SCAN_SORTED, gpu.SCAN_PRUNED):
        gpu.table_set_scan(t, mode)
        br, s = gpu.score_orders(t, orders)
        for b in range(len(orders)):
            assert np.array_equal(br[b], ref[b][1]) and s[b] == ref[b][0], (mode, b)
