"""The native call path of gemm and dot_batch leaves the interpreter to other threads while it is in the library."""
import ctypes
import subprocess
import threading
import time

import pytest
import torch

pytestmark = pytest.mark.gpu

SLOW = r"""
#include <unistd.h>
extern "C" int slow() { usleep(500000); return 0; }     /* a library call that waits, for a full launch queue say */
"""


def test_other_threads_run_during_a_call(tmp_path):
    from paper_2511_10909_b200 import mmasim
    (tmp_path / "slow.cpp").write_text(SLOW)
    subprocess.run(["g++", "-shared", "-fPIC", str(tmp_path / "slow.cpp"), "-o", str(tmp_path / "slow.so")], check=True)
    slow = ctypes.CDLL(str(tmp_path / "slow.so")).slow
    address = lambda f: ctypes.cast(f, ctypes.c_void_p).value
    lib, fast = mmasim._lib, mmasim._fast or mmasim._load_fast()
    model = mmasim.Model("hopper", "fp16", "fp32")
    A = torch.zeros((16, 16), dtype=torch.int16, device="cuda")
    torch.cuda.synchronize()
    fast.bind(address(slow), address(slow), address(lib.mmasim_model_info))
    try:
        for call in (lambda: mmasim.gemm(model, A, A), lambda: mmasim.dot_batch(model, A, A)):
            worker, ticks, t0 = threading.Thread(target=call), 0, time.perf_counter()
            worker.start()
            while worker.is_alive():
                ticks += 1
                time.sleep(0.002)
            assert time.perf_counter() - t0 > 0.45 and ticks > 25, ticks
    finally:
        fast.bind(address(lib.mmasim_gemm_ex), address(lib.mmasim_dot_batch), address(lib.mmasim_model_info))
