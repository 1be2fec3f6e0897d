"""The sum-based score of more orders than one grid of a scan takes (65,535 x 256): every
order's score equals that of the same order in a small call, bit for bit, on either side of the
seam, in the default scan, on a table without sorted parent sets (k > 4) and a pruned one."""
import itertools

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,k,pruned", [(2, 1, False), (2, 1, True), (6, 5, False)])
def test_more_orders_than_a_grid(gpu, n, k, pruned):
    import torch
    import oracle
    B = 65535 * 256 + 300
    rng = np.random.default_rng(3)
    t = gpu.table_from_scores(rng.normal(-2.0, 1.0, (n, oracle.num_sets(n - 1, k))), k)
    if pruned:
        gpu.table_set_scan(t, gpu.SCAN_PRUNED)
    perms = torch.tensor(list(itertools.permutations(range(n))), dtype=torch.uint8, device="cuda")
    few, terms = gpu.score_orders_sum(t, perms)
    g = torch.Generator(device="cuda").manual_seed(1)
    pick = torch.randint(0, len(perms), (B,), generator=g, device="cuda")
    score, node = gpu.score_orders_sum(t, perms[pick])
    assert torch.equal(score, few[pick]) and torch.equal(node, terms[pick])
