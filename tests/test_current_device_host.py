"""A context's work goes to the context's device whatever device is current
when it is asked for: the host code (csrc/runtime.cu) is compiled against a
stand-in of the CUDA runtime with two devices that checks, at every launch,
that the stream belongs to the device that is current. No GPU is used."""
import os
import subprocess

import pytest

from conftest import ROOT

CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

FAKE = r"""
#include <cuda_runtime.h>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "mocd.h"
#include "mocd_internal.h"

struct CUstream_st { int dev; bool capturing; };
static int g_dev = 0, g_wrong = 0, g_launches = 0, g_captures = 0;
static int g_word;  // what opaque handles point to
template <class T> static T handle() { return reinterpret_cast<T>(&g_word); }
static cudaError_t launched(cudaStream_t s)
{
    ++g_launches;
    g_wrong += s->dev != g_dev;
    return cudaSuccess;
}

extern "C" {
cudaError_t cudaSetDevice(int d) { g_dev = d; return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = g_dev; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 4; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = handle<cudaEvent_t>(); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 0; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *) { *p = handle<cudaMemPool_t>(); return cudaSuccess; }
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolGetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t, cudaStream_t) { *p = calloc(n, 1); return cudaSuccess; }
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaStreamCreateWithPriority(cudaStream_t *s, unsigned, int) { *s = new CUstream_st{g_dev, false}; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return cudaStreamCreateWithPriority(s, 0, 0); }
cudaError_t cudaStreamDestroy(cudaStream_t s) { delete s; return cudaSuccess; }
cudaError_t cudaStreamGetPriority(cudaStream_t, int *p) { *p = 0; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) { s->capturing = true; ++g_captures; return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t *g) { s->capturing = false; *g = handle<cudaGraph_t>(); return cudaSuccess; }
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t s, cudaStreamCaptureStatus *st, unsigned long long *, cudaGraph_t *,
                                     const cudaGraphNode_t **deps, const cudaGraphEdgeData **data, size_t *n)
{
    static cudaGraphNode_t none;
    *st = s->capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    if (deps) *deps = &none;
    if (data) *data = nullptr;
    if (n) *n = 0;
    return cudaSuccess;
}
cudaError_t cudaStreamUpdateCaptureDependencies(cudaStream_t, cudaGraphNode_t *, const cudaGraphEdgeData *, size_t, unsigned) { return cudaSuccess; }
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) { *x = handle<cudaGraphExec_t>(); return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphGetNodes(cudaGraph_t, cudaGraphNode_t *, size_t *n) { *n = 0; return cudaSuccess; }
cudaError_t cudaGraphNodeGetType(cudaGraphNode_t, cudaGraphNodeType *t) { *t = cudaGraphNodeTypeEmpty; return cudaSuccess; }
}

namespace mocd {
cudaError_t launch_front(const GenParams &, const PopState &, cudaStream_t s) { return launched(s); }
cudaError_t launch_rows(int, const int32_t *, const int32_t *, const int32_t *, int32_t *, int32_t *, int, const int2 *, int4 *, int4 *, int, cudaStream_t s) { return launched(s); }
cudaError_t launch_select(const GenParams &, const PopState &, int, cudaStream_t s, uint32_t) { return launched(s); }
cudaError_t launch_select_multi(const GenParams *, const PopState *, int, int, cudaStream_t s) { return launched(s); }
cudaError_t launch_evaluate(int, int, int, bool, const int32_t *, const int32_t *, const int32_t *, const int32_t *, uint32_t *, unsigned long long *, unsigned long long *, int, cudaStream_t s, const int32_t *) { return launched(s); }
cudaError_t launch_evaluate_multi(const BatchMember *, const int *, int, int, cudaStream_t s) { return launched(s); }
cudaError_t launch_evaluate_offspring(int, int, int, const int32_t *, const int32_t *, const int32_t *, uint32_t *, unsigned long long *, int, cudaStream_t s, const int32_t *) { return launched(s); }
cudaError_t launch_mutation(const GenParams &, const PopState &, const int4 *, const int4 *, const MutationShape &, cudaStream_t s) { return launched(s); }
cudaError_t launch_crossover(const GenParams &, const PopState &, int, cudaStream_t s) { return launched(s); }
cudaError_t launch_crossover_multi(const BatchMember *, const int *, int, int, int, int, cudaStream_t s) { return launched(s); }
cudaError_t launch_front_stats(const GenParams &, const PopState &, const int32_t *, int, const int32_t *, const int32_t *, const int32_t *, int32_t *, unsigned long long *, uint32_t *, unsigned long long *, unsigned long long *, int, cudaStream_t s) { return launched(s); }
cudaError_t launch_to_node_major(int, int, int, const int32_t *, int32_t *, int *, cudaStream_t s) { return launched(s); }
cudaError_t launch_symmetry_check(int, const int32_t *, const int32_t *, int *, int, cudaStream_t s) { return launched(s); }
cudaError_t launch_init_population(const GenParams &, int, const int32_t *, const int32_t *, int32_t *, cudaStream_t s) { return launched(s); }
cudaError_t launch_gather_individuals(int, int, int, const int32_t *, const int32_t *, const int32_t *, int, int32_t *, cudaStream_t s) { return launched(s); }
cudaError_t check_record_eval(unsigned long long *, bool) { return cudaSuccess; }
cudaError_t check_record_variation(unsigned long long *, bool) { return cudaSuccess; }
size_t stats_acc_words() { return 1; }
int grid_for_hubs(int sms, int) { return sms; }
int grid_for_mutation(int sms, int, int, int, int, int) { return sms; }
int grid_for_crossover(int sms, int, int) { return sms; }
int grid_for_eval_intra(int sms) { return sms; }
int crossover_row_words(int) { return 1; }
int mutation_warps_per_block() { return 4; }
bool evaluate_needs_histogram(int64_t, int, bool) { return false; }
}

#define DO(call) if (const int rc = (call)) { printf("%s: %d\n", #call, rc); return 1; }

int main()
{
    const int64_t rp[5] = {0, 2, 4, 6, 8};  // a ring of four nodes
    const int32_t ci[8] = {1, 3, 0, 2, 1, 3, 0, 2};
    mocd_params p = {};
    p.pop_size = 4;
    p.n_parents = 2;
    p.p_crossover = 0.8;
    p.p_mutation = 0.2;
    for (int own = 0; own < 2; ++own) {
        // One context per device; a context with a caller's stream, then one with its own.
        mocd_ctx *c[2];
        for (int d = 0; d < 2; ++d) {
            cudaSetDevice(d);
            CUstream_st *s = own ? nullptr : new CUstream_st{d, false};
            DO(mocd_graph_upload(&c[d], 4, rp, ci, s));
            DO(mocd_population_init(c[d], &p));
        }
        // Device 1 is current. Each call captures a graph of context 0.
        const int before = g_captures;
        DO(mocd_generation(c[0], 40));
        if (g_captures != before + 1) { printf("the long run captured %d graphs\n", g_captures - before); return 1; }
        DO(mocd_set_timing(c[0], 1));
        DO(mocd_generation(c[0], 1));
        if (g_captures != before + 2) { printf("the timed run captured nothing\n"); return 1; }
        if (g_dev != 1) { printf("the caller's device changed to %d\n", g_dev); return 1; }
        for (int d = 0; d < 2; ++d) { cudaSetDevice(d); mocd_destroy(c[d]); }
    }
    printf("%d of %d launches on another device's stream\n", g_wrong, g_launches);
    return g_wrong != 0;
}
"""


def test_graphs_are_captured_on_the_contexts_device(tmp_path):
    if not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    fake, exe = tmp_path / "fake.cpp", tmp_path / "fake"
    fake.write_text(FAKE)
    csrc = os.path.join(ROOT, "paper_2506_01752_gb300", "csrc")
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-w", "-I", os.path.join(CUDA, "include"),
                    "-I", os.path.join(ROOT, "include"), "-I", csrc, "-x", "c++",
                    os.path.join(csrc, "runtime.cu"), str(fake), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
