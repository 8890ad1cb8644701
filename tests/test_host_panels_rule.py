"""Which tiles row panels of ragged rows take: the dispatcher's own rule, called on the host, on both sides of its lines (times of both
sides are at the rule)."""
import pytest

from helpers import host_program

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "mmasim_internal.h"
using namespace mmasim;
int main(int, char** argv) {            // arch, input type, accumulator type, M, N, K, row stride, panels, rows of the last
    mmasim_model m;
    const char* why = "";
    if (!registry_lookup(std::atoi(argv[1]), std::atoi(argv[2]), std::atoi(argv[2]), std::atoi(argv[3]), &m, &why)) return 1;
    GemmArgs g;
    std::memset(&g, 0, sizeof(g));
    g.M = std::atoi(argv[4]); g.N = std::atoi(argv[5]); g.K = std::atoi(argv[6]);
    g.lda = g.ldb = std::atoi(argv[7]);
    g.ldc = g.ldd = g.N;
    std::printf("%d %d\n", int(direct_size(m.dev, g)), int(panels_on_large_tiles(m.dev, g, std::atoi(argv[8]), std::atoi(argv[9]))));
}
"""


@pytest.fixture(scope="module")
def ask(tmp_path_factory):
    run = host_program(tmp_path_factory.mktemp("panels"), PROGRAM)
    from paper_2511_10909_b200 import mmasim
    return lambda key, *a: run(mmasim.ARCH[key[0]], mmasim.FMT[key[1]], mmasim.ACC[key[2]], *a)[0].split()


@pytest.mark.parametrize("key,M,N,K,ld,panels,last,large", [
    (("cdna3", "e4m3", "fp32"), 418, 1999, 1552, 1552, 1, 418, 0), (("hopper", "e4m3", "fp32"), 786, 591, 736, 744, 1, 786, 1),          # one panel
    (("ampere", "tf32", "fp32"), 1998, 454, 1556, 1556, 4, 462, 0), (("volta", "fp16", "fp32"), 2459, 3151, 364, 364, 5, 411, 1), (("ampere", "fp16", "fp32"), 2733, 2512, 624, 624, 6, 173, 1),       # several
    (("ampere", "bf16", "fp32"), 1479, 742, 1800, 1800, 3, 455, 0), (("ada", "e5m2", "fp32"), 1219, 935, 1904, 1904, 2, 579, 1),         # places left
    (("ampere", "bf16", "fp32"), 1136, 1247, 744, 744, 3, 112, 0), (("ampere", "fp16", "fp32"), 624, 3300, 520, 520, 2, 112, 1), (("hopper", "e4m3", "fp32"), 1108, 1702, 1248, 1256, 2, 84, 1),        # a short last one
    (("cdna3", "tf32", "fp32"), 1279, 853, 3072, 3072, 3, 255, 1), (("ampere", "fp16", "fp32"), 624, 3300, 544, 544, 2, 112, 1)], ids=str)   # whole chunks
def test_panels_of_ragged_rows(ask, key, M, N, K, ld, panels, last, large):
    none, on_large = ask(key, M, N, K, ld, panels, last)
    assert none == "0"                                      # (one call by itself takes the large tiles)
    assert on_large == str(large)
