"""The integer long division of the crowding distance (csrc/ratio.cuh) as the
GPU runs it, whose reciprocal estimate is another one than the host's: equal to
the IEEE division of the two doubles, bit for bit."""
import os
import subprocess

import pytest

from conftest import ROOT
from paper_2506_01752_gb300 import build as cuda_build

pytestmark = pytest.mark.gpu

SRC = r"""
#include "ratio.cuh"
#include <cstdio>
#include <random>
#include <vector>
__global__ void run(long n, const long long *gap, const long long *range, unsigned long long *bits)
{
    for (long k = blockIdx.x * (long)blockDim.x + threadIdx.x; k < n; k += (long)gridDim.x * blockDim.x)
        bits[k] = mocd::ratio_bits(gap[k], range[k]);
}
int main()
{
    std::vector<long long> gap, range;
    auto add = [&](long long g, long long d) { gap.push_back(g); range.push_back(d); };
    for (long long d = 1; d < 300; ++d)
        for (long long g = 0; g <= d; ++g) add(g, d);
    // around every power of two: significands that round up to the next one
    for (int s = 50; s < 63; ++s)
        for (int i = -20; i < 20; ++i)
            for (int j = -20; j < 20; ++j) {
                const long long d = (1ll << s) + i;
                add((1ll << (s - 3)) + j, d);
                if (j <= i) add((1ll << s) + j, d);
            }
    std::mt19937_64 r(11);
    for (long k = 0; k < 4000000; ++k) {
        long long d = (long long)(r() >> (1 + r() % 63));
        if (d <= 0) d = 1;
        add(k & 1 ? (long long)(r() % ((unsigned long long)d + 1)) : d >> (r() % 62), d);
    }
    const long n = (long)gap.size();
    long long *g, *d;
    unsigned long long *b;
    if (cudaMallocManaged(&g, 8 * n) || cudaMallocManaged(&d, 8 * n) || cudaMallocManaged(&b, 8 * n)) return 2;
    for (long k = 0; k < n; ++k) { g[k] = gap[k]; d[k] = range[k]; b[k] = ~0ull; }
    run<<<1024, 256>>>(n, g, d, b);
    if (cudaDeviceSynchronize() != cudaSuccess) return 2;
    long bad = 0;
    for (long k = 0; k < n; ++k) {
        const double x = (double)gap[k] / (double)range[k];
        unsigned long long want;
        memcpy(&want, &x, 8);
        bad += want != b[k];
    }
    printf("%ld of %ld\n", bad, n);
    return bad != 0;
}
"""


def test_ratio_on_the_device_equals_ieee_division(tmp_path):
    src, exe = tmp_path / "ratio.cu", tmp_path / "ratio"
    src.write_text(SRC)
    subprocess.run([cuda_build._nvcc(), *cuda_build.ARCH, *cuda_build.FLAGS, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
