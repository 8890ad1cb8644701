"""mmasim_gemm_host in one panel, in several, and with a last panel shorter than the others, from several threads at once and after the
kept streams were given back, and with D over the memory of an operand, against the same product on device memory."""
import threading

import numpy as np
import pytest
import torch

from paper_2511_10909_b200 import workloads as wl

pytestmark = pytest.mark.gpu
gu = pytest.importorskip("gpu_util") if torch.cuda.is_available() else None


def test_more_calls_at_once_than_sets_of_streams_are_kept():
    """Ten calls at a time, twice, with the kept ones given back in between."""
    from paper_2511_10909_b200 import mmasim
    key, (M, N, K) = ("ampere", "fp16", "fp32"), (100, 90, 48)
    inp = wl.normal_inputs(key[1], key[2], M, N, K, seed=7)
    want = gu.run_gemm(key, inp)
    model = mmasim.Model(*key)
    for _ in range(2):
        got = [None] * 10
        gate = threading.Barrier(len(got))

        def call(i):
            gate.wait()
            got[i] = mmasim.gemm_host(model, inp["A"], inp["B"], inp["C"])
        threads = [threading.Thread(target=call, args=(i,)) for i in range(len(got))]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert all(np.array_equal(x, want) for x in got)
        mmasim.host_release()


@pytest.mark.parametrize("key,shape", [(("hopper", "e4m3", "fp32"), (2100, 1100, 256)), (("ampere", "bf16", "fp32"), (1500, 1300, 40)),
                                       (("hopper", "fp16", "fp32"), (513, 6000, 64)), (("blackwell", "nvf4", "fp32"), (1700, 1600, 128)),
                                       (("volta", "fp16", "fp16"), (40, 30, 20))], ids=str)
def test_panels_and_threads(key, shape):
    from paper_2511_10909_b200 import mmasim
    M, N, K = shape
    inp = wl.normal_inputs(key[1], key[2], M, N, K, seed=5)
    want = gu.run_gemm(key, inp)
    model = mmasim.Model(*key)
    got = [None] * 3

    def call(i):
        got[i] = mmasim.gemm_host(model, inp["A"], inp["B"], inp["C"], K=K, sfa=inp.get("sfa"), sfb=inp.get("sfb"))
    threads = [threading.Thread(target=call, args=(i,)) for i in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for x in got:
        assert np.array_equal(x.view(want.dtype), want)
    mmasim.host_release()
    call(0)
    assert np.array_equal(got[0].view(want.dtype), want)


def test_output_over_an_operand():
    """D in the place of C, one row further, and over the second half of A's rows: the words of the product of what was there before."""
    from paper_2511_10909_b200 import mmasim
    key, (M, N, K) = ("hopper", "e4m3", "fp32"), (1024, 1024, 2048)
    inp = wl.normal_inputs(key[1], key[2], M, N, K, seed=6)
    want = gu.run_gemm(key, inp)
    model = mmasim.Model(*key)
    for shift in (0, 1):
        buf = np.zeros((M + 1, N), dtype=np.uint32)
        buf[:M] = inp["C"]
        got = mmasim.gemm_host(model, inp["A"], inp["B"], buf[:M], out=buf[shift:M + shift])
        assert np.array_equal(got, want), shift
    half = M * K // 2
    flat = np.zeros(half + 4 * M * N, dtype=np.uint8)
    A = flat[:M * K].reshape(M, K)
    A[:] = inp["A"]
    got = mmasim.gemm_host(model, A, inp["B"], inp["C"], out=flat[half:].view(np.uint32).reshape(M, N))
    assert np.array_equal(got, want)


@pytest.mark.parametrize("key,shape,variant", [(("ampere", "tf32", "fp32"), (1998, 454, 1556), "small_tiles"), (("ampere", "bf16", "fp32"), (1136, 1247, 744), "small_tiles"),
                                               (("ada", "e5m2", "fp32"), (1726, 527, 1712), "large_tiles")], ids=str)
def test_panels_of_ragged_rows(key, shape, variant):
    from paper_2511_10909_b200 import mmasim
    M, N, K = shape
    inp = wl.normal_inputs(key[1], key[2], M, N, K, seed=8)
    want = gu.run_gemm(key, inp)
    got = mmasim.gemm_host(mmasim.Model(*key), inp["A"], inp["B"], inp["C"])
    assert mmasim.last_variant() == variant
    assert np.array_equal(got.view(want.dtype), want)
