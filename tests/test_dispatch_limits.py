"""Where the kernels whose offsets inside a row are 32-bit end: the dispatcher's own predicates, called on the host, at the row lengths
on both sides of the limit (2 GiB rows; 2^21 chunks for the kernels that tag a chunk's number in 21 bits)."""
import pytest

from helpers import host_program

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "mmasim_internal.h"
using namespace mmasim;
int main(int argc, char** argv) {       // arch, input type, accumulator type, then K ...
    mmasim_model m;
    const char* why = "";
    if (!registry_lookup(std::atoi(argv[1]), std::atoi(argv[2]), std::atoi(argv[2]), std::atoi(argv[3]), &m, &why)) return 1;
    for (int i = 4; i < argc; ++i) {
        GemmArgs g;
        std::memset(&g, 0, sizeof(g));
        g.M = g.N = 2;
        g.K = std::atoll(argv[i]);
        g.lda = g.ldb = g.K;
        g.ldc = g.ldd = 2;
        const bool small = direct_size(m.dev, g) != DIRECT_NONE;
        g.N = 1;
        g.dot_mode = 1;
        std::printf("%d %d\n", int(small), int(dot_stream_supported(m.dev, g)));
    }
}
"""


@pytest.fixture(scope="module")
def ask(tmp_path_factory):
    run = host_program(tmp_path_factory.mktemp("limits"), PROGRAM)
    from paper_2511_10909_b200 import mmasim
    return lambda key, *K: [tuple(x == "1" for x in line.split())
                            for line in run(mmasim.ARCH[key[0]], mmasim.FMT[key[1]], mmasim.ACC[key[2]], *K)]


# bytes per element; the largest K of the small-tile kernels, if it is not that of 2 GiB rows
@pytest.mark.parametrize("key,size,last", [(("ampere", "tf32", "fp32"), 4, None), (("ampere", "bf16", "fp32"), 2, None), (("volta", "fp16", "fp16"), 2, None),
                                           (("hopper", "e4m3", "fp32"), 1, None), (("cdna3", "fp16", "fp32"), 2, None),
                                           (("cdna3", "bf16", "fp32"), 2, 2 ** 26), (("cdna3", "tf32", "fp32"), 4, 2 ** 26),
                                           (("cdna2", "fp16", "fp32"), 2, 0)], ids=str)
def test_row_length_limits(ask, key, size, last):
    rows = 2 ** 31 // size                                  # elements of a 2 GiB row
    first = rows if last is None else last
    before, at, beyond = ask(key, max(first - 4096, 32), max(first, 32), 4 * rows)
    assert before[0] == (first > 0) and not at[0] and not beyond[0], (key, before, at, beyond)
    before, at, beyond = ask(key, rows - 1024, rows, 4 * rows)
    assert before[1] and not at[1] and not beyond[1], (key, before, at, beyond)
