"""The integer long division of the crowding distance (csrc/ratio.cuh) equals
the IEEE division of the two doubles, bit for bit."""
import os
import subprocess

from conftest import ROOT

SRC = r"""
#include "ratio.cuh"
#include <cstdio>
#include <random>
static long bad = 0;
static void check(int64_t gap, int64_t range)
{
    const double x = (double)gap / (double)range;
    uint64_t bits;
    memcpy(&bits, &x, 8);
    bad += bits != mocd::ratio_bits(gap, range);
}
int main()
{
    std::mt19937_64 r(7);
    for (int64_t d = 1; d < 300; ++d)
        for (int64_t g = 0; g <= d; ++g) check(g, d);
    // around every power of two: significands that round up to the next one
    for (int s = 50; s < 63; ++s)
        for (int i = -20; i < 20; ++i)
            for (int j = -20; j < 20; ++j) {
                const int64_t d = (1ll << s) + i;
                check((1ll << (s - 3)) + j, d);
                if (j <= i) check((1ll << s) + j, d);
            }
    for (long k = 0; k < 4000000; ++k) {
        int64_t d = (int64_t)(r() >> (1 + r() % 63));
        if (d <= 0) d = 1;
        const int64_t g = k & 1 ? (int64_t)(r() % ((uint64_t)d + 1)) : d >> (r() % 62);
        check(g, d);
    }
    printf("%ld\n", bad);
    return bad != 0;
}
"""


def test_ratio_equals_ieee_division(tmp_path):
    src = tmp_path / "ratio.cpp"
    src.write_text(SRC)
    exe = tmp_path / "ratio"
    csrc = os.path.join(ROOT, "paper_2506_01752_gb300", "csrc")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", csrc, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
