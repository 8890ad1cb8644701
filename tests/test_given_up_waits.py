"""Calls that wait for their kernels report bounded waits that ran out: the status, the message and the total, from counts that the test
makes up on the host (no kernel is made to wait in vain)."""
import re

from helpers import host_program

PROGRAM = r"""
#include <cstdio>
#include "mmasim_internal.h"
using namespace mmasim;
int main() {
    set_error("as before");
    std::printf("%d %s\n", given_up_waits(MMASIM_OK, 0u, 0, "call"), mmasim_last_error());
    std::printf("%d ", given_up_waits(MMASIM_ERR_SHAPE, 2u, 0, "call"));
    std::printf("%s\n", mmasim_last_error());
    std::printf("%d ", given_up_waits(MMASIM_OK, 3u, 0, "call"));
    std::printf("%s\n", mmasim_last_error());
    std::printf("%d\n", given_up_waits(MMASIM_OK, 1u, -1, "call"));
}
"""


def test_status_and_message(tmp_path):
    assert host_program(tmp_path, PROGRAM)() == [
        "0 as before", "3 as before", "6 call: 3 CTAs gave up waiting for a bulk copy and stored nothing", "6"]


def test_both_synchronous_calls_ask():
    """mmasim_gemm_host and mmasim_deviation_stats hand their kernels the call's own counter and return what it says."""
    import os
    from paper_2511_10909_b200.build import CSRC
    text = open(os.path.join(CSRC, "mmasim_api.cpp")).read()
    for call in ("mmasim_gemm_host", "mmasim_deviation_stats"):
        body = re.search(r"\nint %s\(.*?\n}\n" % call, text, flags=re.S).group(0)
        assert "g.copy_timeouts = lane.gave_up_dev" in body and f'given_up_waits(st, count, device, "{call}")' in body, call
