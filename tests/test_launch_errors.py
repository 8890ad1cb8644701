"""A launch that fails is the error of its call: nothing stays behind in the thread for the next caller that asks the runtime (torch asks
after every launch of its own).  The launchers are called on the host, the runtime's launch and its record of the last error are
stand-ins of the program: nothing reaches a GPU."""
from helpers import host_program

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include <cuda_runtime.h>
#include "mmasim_internal.h"
using namespace mmasim;
// in front of the runtime's own functions of these names
static cudaError_t last = cudaSuccess;
extern "C" __attribute__((visibility("default"))) cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**) { return last = cudaErrorInvalidConfiguration; }
extern "C" __attribute__((visibility("default"))) cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
extern "C" __attribute__((visibility("default"))) cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
int main() {
    mmasim_model m;
    const char* why = "";
    if (!registry_lookup(MMASIM_HOPPER, MMASIM_F16, MMASIM_F16, MMASIM_ACC_F32, &m, &why)) return 1;
    GemmArgs g;
    std::memset(&g, 0, sizeof(g));
    g.M = 64; g.N = 1; g.K = 16;
    g.lda = g.ldb = 16; g.ldc = g.ldd = 1;
    g.dot_mode = 1;
    std::printf("%d", launch_dot_stream(m.dev, g, nullptr));
    std::printf(" %d\n", int(last));
    std::printf("%d", launch_generic(m.dev, g, nullptr));
    std::printf(" %d\n", int(last));
    std::printf("%d", launch_error_stats(ACC_F32, 64, nullptr, nullptr, nullptr, nullptr));
    std::printf(" %d\n", int(last));
}
"""


def test_a_failed_launch_leaves_no_error_behind(tmp_path):
    assert host_program(tmp_path, PROGRAM)() == ["5 0"] * 3         # MMASIM_ERR_CUDA, cudaSuccess
