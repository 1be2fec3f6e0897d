"""Per-context set-up when threads meet at it: whichever thread comes first, none returns
before the set-up is done (a kernel launched before its shared-memory attribute is set is
refused), it runs once per context and device, and again after a failure."""
import os
import subprocess
import sys

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1210_5128_gb300", "csrc")

PROGRAM = r"""
#include "bn_once.cuh"
#include <atomic>
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>
int main()
{
    int bad = 0;
    for (int round = 0; round < 20; ++round) {
        static bn::ContextOnce once;
        const unsigned long long id = 100 + round;
        std::atomic<int> set{0}, runs{0}, early{0};
        std::vector<std::thread> th;
        for (int t = 0; t < 8; ++t)
            th.emplace_back([&] {
                const int rc = once.run(3, id, [&] {
                    ++runs;
                    std::this_thread::sleep_for(std::chrono::milliseconds(5));
                    set = 1;
                    return 0;
                });
                if (rc != 0 || !set) ++early;
            });
        for (auto& x : th) x.join();
        bad += early != 0;
        bad += runs != 1;
    }
    bn::ContextOnce o;
    int n = 0;
    auto f = [&] { return ++n == 1 ? -7 : 0; };
    bad += o.run(0, 5, f) != -7 || n != 1;            // a failure is reported and tried again
    bad += o.run(0, 5, f) != 0 || n != 2;
    bad += o.run(0, 5, f) != 0 || n != 2;
    bad += o.run(1, 5, f) != 0 || n != 3;             // another device
    bad += o.run(0, 6, f) != 0 || n != 4;             // another context
    bad += o.run(0, 0, f) != 0 || n != 5;             // no name: every time
    bad += o.run(0, 0, f) != 0 || n != 6;
    bad += o.run(64, 5, f) != 0 || n != 7;
    bad += o.run(-1, 5, f) != 0 || n != 8;
    printf("%d\n", bad);
    return bad != 0;
}
"""


def test_no_thread_passes_an_unfinished_set_up(tmp_path):
    (tmp_path / "t.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-pthread", "-x", "c++", "-I", CSRC, "-o", str(tmp_path / "t"),
                    str(tmp_path / "t.cpp")], check=True)
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


THREADS = r"""
import sys
import threading
import numpy as np
sys.path.insert(0, sys.argv[1])
import paper_1210_5128_gb300 as bn
rng = np.random.default_rng(1)
# sizes that need different shared memory: rows, cells of a count table, sets a node
nets = [((rng.random((m, n)) * a).astype(np.uint8), np.full(n, a, np.uint8), k)
        for m, n, a, k in [(5000, 12, 4, 5), (40, 20, 2, 4), (900, 24, 3, 4), (64, 6, 2, 2)] * 2]
orders = [np.stack([rng.permutation(x.shape[1]) for _ in range(5)]).astype(np.uint8) for x, _, _ in nets]
out = [None] * len(nets)
go = threading.Barrier(len(nets))

def work(i):
    x, a, k = nets[i]
    go.wait()
    try:
        t = bn.build_scores(x, a, k)
        bn.table_set_scan(t, bn.SCAN_PRUNED)
        out[i] = (bn.table_scores(t), bn.score_orders(t, orders[i])[1])
    except Exception as e:
        out[i] = e

th = [threading.Thread(target=work, args=(i,)) for i in range(len(nets))]
[t.start() for t in th]
[t.join() for t in th]
for (x, a, k), o, r in zip(nets, orders, out):
    assert isinstance(r, tuple), r
    t = bn.build_scores(x, a, k)
    assert np.array_equal(bn.table_scores(t), r[0]) and np.array_equal(bn.score_orders(t, o)[1], r[1])
"""


@pytest.mark.gpu
def test_first_calls_of_a_process_from_threads(gpu):
    root = os.path.dirname(os.path.dirname(CSRC))
    for _ in range(3):
        r = subprocess.run([sys.executable, "-c", THREADS, root], capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
