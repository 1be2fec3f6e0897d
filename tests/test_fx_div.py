"""A table entry's rounding and division by ln 10 in integers, bit for bit against the same
steps in FP64: low word to 53 bits, sum, quotient, each rounded to nearest.  Sums of every
magnitude and sign, carries out of the low word, ties, and zero."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1210_5128_gb300", "csrc")

PROGRAM = r"""
#include "bn_fx.cuh"
#include <cstdio>
#include <cstring>
#include <random>
static uint64_t fp64(int64_t hi, uint64_t lo)
{
    volatile double l = (double)lo;
    l = l * 0x1p-64;
    volatile double x = (double)hi + l;
    const double q = x / 2.302585092994045684017991454684364208;
    uint64_t b;
    memcpy(&b, &q, 8);
    return b;
}
int main(int, char** argv)
{
    const int kind = atoi(argv[1]);
    std::mt19937_64 g(kind);
    long bad = 0, n = 0;
    auto check = [&](int64_t hi, uint64_t lo) {
        bad += bn::fx_div_ln10(((unsigned __int128)(uint64_t)hi << 64) | lo) != fp64(hi, lo);
        ++n;
    };
    for (int64_t hi = -3; hi <= 3; ++hi)
        for (int b = 0; b < 64; ++b)
            for (uint64_t d = -5; d != 6; ++d) {
                check(hi, ((uint64_t)1 << b) + d);
                check(hi << (b % 50), d);
            }
    for (int i = 0; i < 4000000; ++i) {
        int64_t hi = ((int64_t)g() >> 12) >> (g() % 52);
        uint64_t lo = g();
        if (kind == 1) lo >>= g() % 64;
        if (kind == 2) lo &= ~(uint64_t)0 << (g() % 64);
        if (kind == 3) lo = ~(lo >> (g() % 64)), hi = g() % 2 ? hi : -(int64_t)(g() % 2);
        check(hi, lo);
    }
    printf("%ld of %ld\n", bad, n);
    return bad != 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    (d / "t.cpp").write_text("#include <cstdlib>\n" + PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC, "-o", str(d / "t"), str(d / "t.cpp")],
                   check=True)
    return str(d / "t")


@pytest.mark.parametrize("kind", [0, 1, 2, 3])
def test_division_matches_fp64(program, kind):
    r = subprocess.run([program, str(kind)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
