"""The sum score's power of ten in 59-bit fixed point against the C library's in long double:
every value within 2^-55 of itself, over the whole decade, near its ends and where the table
digits change, and no bias above a quarter of that."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1210_5128_gb300", "csrc")

PROGRAM = r"""
#include "bn_fx.cuh"
#include <cmath>
#include <cstdio>
#include <random>
static const bn::Exp2Tables T = bn::make_exp2();
int main()
{
    std::mt19937_64 g(1);
    long double worst = 0, sum = 0;
    long n = 0;
    auto check = [&](uint64_t d) {
        if (d > (uint64_t)1 << 60) return;
        const long double e = exp2l(59 - ldexpl((long double)d, -60) * 3.321928094887362347870319429489390175865L);
        const long double r = ((long double)bn::exp10_fx(d, T.v) - e) / e;
        worst = fmaxl(worst, fabsl(r));
        sum += r;
        ++n;
    };
    const uint64_t one = (uint64_t)1 << 60;
    if (bn::exp10_fx(0, T.v) != ((uint64_t)1 << 59) - 1) return 2;       // 32 of the largest fit 64 bits
    for (uint64_t i = 0; i < 2000; ++i) check(i), check(one - i);
    // around whole digits of d log2 10 in 1/64, 1/4096 and 1/262144
    for (int t = 1; t <= 3; ++t)
        for (int i = 0; i < 20000; ++i) {
            const uint64_t dig = g() % ((uint64_t)3322 << (6 * t) >> 10);
            const uint64_t d = (uint64_t)(ldexpl((long double)dig, 60 - 6 * t) / 3.321928094887362347870319429489390175865L);
            check(d + g() % 65 - 32);
        }
    for (int i = 0; i < 2000000; ++i) check(g() & (one - 1));
    printf("worst 2^%.3f mean %.3f 2^-55\n", (double)log2l(worst), (double)(sum / n * 0x1p55L));
    return !(worst <= 0x1p-55L && fabsl(sum / n) <= 0x1p-57L);
}
"""


def test_power_of_ten(tmp_path):
    (tmp_path / "t.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", CSRC, "-o", str(tmp_path / "t"), str(tmp_path / "t.cpp")], check=True)
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    print(r.stdout)
