"""Where a call of ragged rows goes that may not have scratch: to the small tiles, when the allocation fails and when its stream is being
recorded into a graph; whole chunks are refused without memory, and allocate in a graph.  The launcher is called on the host with stand-ins
for the runtime's functions: nothing reaches a GPU."""
import pytest

from helpers import host_program

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <cuda_runtime.h>
#include "mmasim_internal.h"
using namespace mmasim;
static int launches = 0, allocations = 0;
static bool memory = true, recording = false;
#define STANDIN extern "C" __attribute__((visibility("default"))) cudaError_t
STANDIN cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**) { ++launches; return cudaSuccess; }
STANDIN cudaGetLastError() { return cudaSuccess; }
STANDIN cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
STANDIN cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
STANDIN cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) { *p = reinterpret_cast<cudaMemPool_t>(64); return cudaSuccess; }
STANDIN cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
STANDIN cudaMallocFromPoolAsync(void** p, size_t, cudaMemPool_t, cudaStream_t) { if (!memory) return cudaErrorMemoryAllocation; ++allocations; *p = reinterpret_cast<void*>(4096); return cudaSuccess; }
STANDIN cudaFreeAsync(void*, cudaStream_t) { return cudaSuccess; }
STANDIN cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) { *s = recording ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone; return cudaSuccess; }
int main(int, char** argv) {            // arch, input type, accumulator type, K, row stride of A, memory, recording
    mmasim_model m;
    const char* why = "";
    if (!registry_lookup(std::atoi(argv[1]), std::atoi(argv[2]), std::atoi(argv[2]), std::atoi(argv[3]), &m, &why)) return 1;
    GemmArgs g;
    std::memset(&g, 0, sizeof(g));
    g.M = g.N = 1024;
    g.K = g.ldb = std::atoi(argv[4]);
    g.lda = std::atoi(argv[5]);
    g.ldc = g.ldd = 1024;
    memory = std::atoi(argv[6]);
    recording = std::atoi(argv[7]);
    const int st = launch_fast_tfdpa(m.dev, g, nullptr);
    std::printf("%d %d %d %s\n", st, launches, allocations, mmasim_last_variant());
}
"""


@pytest.fixture(scope="module")
def route(tmp_path_factory):
    run = host_program(tmp_path_factory.mktemp("routes"), PROGRAM)
    from paper_2511_10909_b200 import mmasim
    def ask(key, K, lda, memory=1, recording=0):
        status, launches, allocations, variant = run(mmasim.ARCH[key[0]], mmasim.FMT[key[1]], mmasim.ACC[key[2]], K, lda, memory, recording)[0].split()
        return int(status), int(launches), int(allocations), variant
    return ask


@pytest.mark.parametrize("key", [("ampere", "fp16", "fp32"), ("hopper", "e4m3", "fp32"), ("ada", "e5m2", "fp16"), ("blackwell", "e4m3", "fp32"), ("cdna3", "e4m3", "fp32"),
                                 ("cdna3", "bf16", "fp32"), ("cdna1", "bf16", "fp32")], ids="-".join)
def test_ragged_rows_without_scratch(route, key):
    large, small = (0, 2, 1, "large_tiles"), (0, 1, 0, "small_tiles")       # decode and product; one kernel
    for K, lda in ((992 if key[1] == "bf16" else 1024, 1031), (1008, 1008) if key != ("blackwell", "e4m3", "fp32") else (1024, 1025)):
        assert route(key, K, lda) == large
        assert route(key, K, lda, memory=0) == small
        assert route(key, K, lda, recording=1) == small
    assert route(key, 1024, 1024) == route(key, 1024, 1024, recording=1) == large
    status, launches, allocations, variant = route(key, 1024, 1024, memory=0)
    assert (status, launches, allocations) == (5, 0, 0)
