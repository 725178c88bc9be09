"""A refused launch is an error of the call, not a result that was never
written: the scoring's host code (csrc/k_eval.cu, csrc/noalloc.cu) is linked
against a stand-in of the CUDA runtime that refuses one call of its choice. No
GPU is used."""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT
from paper_2506_01752_gb300 import build as cuda_build

FAKE = r"""
#include <cuda_runtime_api.h>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "mocd.h"

static int g_refuse = -1, g_call = 0;
static cudaError_t g_last = cudaSuccess;
static cudaError_t call()
{
    if (g_call++ != g_refuse) return cudaSuccess;
    return g_last = cudaErrorInvalidValue;
}
static dim3 g_grid, g_block;
static size_t g_shared;
static void *g_stream;

extern "C" {
// What the compiler's launch code calls.
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, void *, void *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t n, void *s)
{
    g_grid = g; g_block = b; g_shared = n; g_stream = s;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *n, void *s)
{
    *g = g_grid; *b = g_block; *n = g_shared; *(void **)s = g_stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void **, size_t, cudaStream_t) { return call(); }
// The runtime.
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *, void **) { return call(); }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return call(); }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return call(); }
cudaError_t cudaGetLastError() { const cudaError_t e = g_last; g_last = cudaSuccess; return e; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 4; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *) { static int scratch; *p = &scratch; return cudaSuccess; }
}

int main(int argc, char **argv)
{
    const int n = atoi(argv[1]), count = atoi(argv[2]);
    const int32_t word = 0;
    int64_t out[2];
    // Once with every call granted, then with each of them refused in turn.
    int calls = 0, bad = 0;
    for (g_refuse = -1; g_refuse < calls || g_refuse == -1; ++g_refuse) {
        g_call = 0;
        const int rc = mocd_evaluate_noalloc(&word, &word, n, &word, count, out, out + 1, nullptr);
        if (g_refuse == -1) calls = g_call;
        if ((rc == MOCD_OK) != (g_refuse == -1)) {
            printf("call %d of %d refused: status %d\n", g_refuse, calls, rc);
            ++bad;
        }
    }
    printf("%d calls\n", calls);
    return bad || calls < 2;
}
"""


def test_every_refused_call_of_the_scoring_is_reported(tmp_path):
    nvcc = cuda_build._nvcc()
    if not shutil.which(nvcc):
        pytest.skip("no nvcc")
    home = os.path.dirname(os.path.dirname(shutil.which(nvcc)))
    src, exe = tmp_path / "fake.cpp", tmp_path / "fake"
    src.write_text(FAKE)
    objs = []
    for name in ("k_eval", "noalloc"):
        objs.append(str(tmp_path / (name + ".o")))
        subprocess.run([nvcc, *cuda_build.ARCH, *cuda_build.FLAGS, "-c",
                        os.path.join(cuda_build.CSRC, name + ".cu"), "-o", objs[-1]], check=True)
    subprocess.run(["g++", "-O1", "-std=c++17", "-w", "-I", os.path.join(home, "include"), "-I",
                    os.path.join(ROOT, "include"), str(src), *objs, "-o", str(exe), "-lpthread"], check=True)
    # Both histogram forms: in shared memory and in the fixed array.
    for n, count in ((1000, 1), (1000, 128), (30_000, 20), (40_960, 100), (40_961, 100), (200_000, 20)):
        out = subprocess.run([str(exe), str(n), str(count)], capture_output=True, text=True)
        assert out.returncode == 0, (n, count, out.stdout)
        # A small scoring costs what it issues: two launches.
        assert n > 1000 or out.stdout == "2 calls\n", (n, count, out.stdout)
