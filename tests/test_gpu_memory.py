"""What the library keeps of the device's memory: at most 2 GiB after a larger table is freed,
and nothing (beyond what driver and kernels took on the way) after release_memory, with live
objects untouched."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
MiB = 1 << 20


def test_freed_memory_goes_back(gpu):
    import torch
    rng = np.random.default_rng(0)

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    x, ar = rng.integers(0, 2, (64, 60)).astype(np.uint8), np.full(60, 2, np.uint8)
    small = gpu.build_scores(x[:, :12], ar[:12], 3)
    orders = np.stack([rng.permutation(12) for _ in range(7)]).astype(np.uint8)
    want = gpu.score_orders(small, orders)
    gpu.build_scores(x, ar, 4).free()                  # every kernel of the build is loaded
    gpu.release_memory()
    before = free()
    tabs = [gpu.build_scores(x, ar, 4) for _ in range(4)]          # 0.7 GB each
    held = sum(gpu.table_info(t)["device_bytes"] for t in tabs)
    assert held > 2400 * MiB and before - free() >= held
    for t in tabs:
        t.free()
    gpu.score_orders(small, orders)                    # (memory above the limit goes at a synchronisation)
    assert before - free() <= 2048 * MiB + 64 * MiB
    gpu.release_memory()
    assert before - free() <= 64 * MiB
    got = gpu.score_orders(small, orders)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
