"""The scratch of mmasim_gemm_host's panels lies in the call's one allocation: what is allocated and freed on the panels' own streams makes
every later allocation look at those streams first.  The call runs on the host with stand-ins for the runtime's functions: nothing reaches
a GPU."""
import pytest

from helpers import host_program

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <cuda_runtime.h>
#include "mmasim_internal.h"
using namespace mmasim;
static int launches = 0, allocations = 0, frees = 0;
static size_t limit = 0, bytes = 0;
static uintptr_t streams = 0;
alignas(256) static unsigned char host_word[256];
#define STANDIN extern "C" __attribute__((visibility("default"))) cudaError_t
STANDIN cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**) { ++launches; return cudaSuccess; }
STANDIN cudaGetLastError() { return cudaSuccess; }
STANDIN cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
STANDIN cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
STANDIN cudaGetSymbolAddress(void** p, const void*) { *p = host_word + 128; return cudaSuccess; }
STANDIN cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) { *p = reinterpret_cast<cudaMemPool_t>(64); return cudaSuccess; }
STANDIN cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
STANDIN cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) {
    if (limit && n > limit) return cudaErrorMemoryAllocation;
    ++allocations; bytes += n; *p = reinterpret_cast<void*>(uintptr_t(1) << 40); return cudaSuccess;
}
STANDIN cudaFreeAsync(void*, cudaStream_t) { ++frees; return cudaSuccess; }
STANDIN cudaHostAlloc(void** p, size_t, unsigned) { *p = host_word; return cudaSuccess; }
STANDIN cudaHostGetDevicePointer(void** p, void* h, unsigned) { *p = h; return cudaSuccess; }
STANDIN cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = reinterpret_cast<cudaStream_t>(++streams << 8); return cudaSuccess; }
STANDIN cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = reinterpret_cast<cudaEvent_t>(++streams << 8); return cudaSuccess; }
STANDIN cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
STANDIN cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
STANDIN cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
STANDIN cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) { *s = cudaStreamCaptureStatusNone; return cudaSuccess; }
STANDIN cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
STANDIN cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
STANDIN cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) { a->type = cudaMemoryTypeHost; return cudaSuccess; }
int main(int, char** argv) {            // arch, input type, accumulator type, M, N, K, bytes that one allocation gets
    mmasim_model* m = mmasim_create_model(std::atoi(argv[1]), std::atoi(argv[2]), std::atoi(argv[3]));
    limit = size_t(std::atoll(argv[7]));
    void* p = reinterpret_cast<void*>(uintptr_t(1) << 41);
    const int st = mmasim_gemm_host(m, std::atoi(argv[4]), std::atoi(argv[5]), std::atoi(argv[6]), p, p, nullptr, reinterpret_cast<void*>(uintptr_t(1) << 42), nullptr);
    std::printf("%d %d %d %d %s\n", st, launches, allocations, frees, *mmasim_last_variant() ? mmasim_last_variant() : "none");
}
"""


@pytest.fixture(scope="module")
def ask(tmp_path_factory):
    run = host_program(tmp_path_factory.mktemp("scratch"), PROGRAM)
    from paper_2511_10909_b200 import mmasim
    def call(key, M, N, K, limit=0):
        status, launches, allocations, frees, variant = run(mmasim.ARCH[key[0]], mmasim.FMT[key[1]], mmasim.ACC[key[2]], M, N, K, limit)[0].split()
        return int(status), int(launches), int(allocations), int(frees), variant
    return call


# large tiles of either kind in several panels, ragged and whole chunks; one panel; small tiles
@pytest.mark.parametrize("key,shape,panels,variant", [(("ampere", "bf16", "fp32"), (2048, 2048, 1024), 4, "large_tiles"), (("hopper", "e4m3", "fp32"), (2048, 2048, 2048), 4, "large_tiles"),
                                                      (("hopper", "e4m3", "fp16"), (2048, 2048, 2048), 4, "large_tiles"), (("ampere", "fp16", "fp32"), (2733, 2512, 624), 6, "large_tiles"),
                                                      (("hopper", "e4m3", "fp32"), (511, 4000, 1024), 1, "large_tiles"), (("ampere", "bf16", "fp32"), (128, 128, 64), 1, "small_tiles")], ids=str)
def test_one_allocation(ask, key, shape, panels, variant):
    each = 2 if variant == "large_tiles" else 1
    assert ask(key, *shape) == (0, panels * each, 1, 1, variant)


def test_panels_take_their_own_scratch_where_one_allocation_is_too_large(ask):
    M, N, K = 2048, 2048, 1024
    operands = 2 * (M + N) * K + 4 * M * N                  # and some 31 MB of decoded blocks for each of four panels
    assert ask(("ampere", "bf16", "fp32"), M, N, K, limit=64 << 20) == (0, 8, 5, 5, "large_tiles")
    assert ask(("ampere", "bf16", "fp32"), M, N, K, limit=operands - 1)[0] == 5
