"""A launch that fails is the error of its call: nothing stays behind in the thread for the next caller that asks the runtime (torch asks
after every launch of its own).  Without a GPU every launch fails, so the launchers are called on the host as they are."""
import pytest

from helpers import host_program

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include <dlfcn.h>
#include <cuda_runtime.h>
#include "mmasim_internal.h"
using namespace mmasim;
// (the runtime that the library has brought into the process)
template <class F> F* runtime(const char* name) { return reinterpret_cast<F*>(dlsym(RTLD_DEFAULT, name)); }
int main() {
    auto count = runtime<cudaError_t(int*)>("cudaGetDeviceCount");
    auto take = runtime<cudaError_t()>("cudaGetLastError");
    auto peek = runtime<cudaError_t()>("cudaPeekAtLastError");
    int devices = 0;
    if (count(&devices) == cudaSuccess && devices > 0) { std::puts("device"); return 0; }
    take();
    mmasim_model m;
    const char* why = "";
    if (!registry_lookup(MMASIM_HOPPER, MMASIM_F16, MMASIM_F16, MMASIM_ACC_F32, &m, &why)) return 1;
    GemmArgs g;
    std::memset(&g, 0, sizeof(g));
    g.M = 64; g.N = 1; g.K = 16;
    g.lda = g.ldb = 16; g.ldc = g.ldd = 1;
    g.dot_mode = 1;
    int st = launch_dot_stream(m.dev, g, nullptr);
    std::printf("dot %d %d\n", st, int(peek()));
    st = launch_error_stats(ACC_F32, 64, nullptr, nullptr, nullptr, nullptr);
    std::printf("stats %d %d\n", st, int(peek()));
}
"""


def test_a_failed_launch_leaves_no_error_behind(tmp_path):
    lines = host_program(tmp_path, PROGRAM)()
    if lines == ["device"]:
        pytest.skip("launches succeed here")
    for line in lines:
        name, status, left = line.split()
        assert int(status) == 5 and int(left) == 0, line
    assert len(lines) == 2
