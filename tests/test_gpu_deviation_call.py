"""mmasim_deviation_stats against the same pipeline in three calls: FP32 and FP16 accumulators, ragged sizes, with and without C."""
import numpy as np
import pytest
import torch

from paper_2511_10909_b200 import workloads as wl

pytestmark = pytest.mark.gpu
gu = pytest.importorskip("gpu_util") if torch.cuda.is_available() else None


@pytest.mark.parametrize("key", [("cdna3", "fp16", "fp32"), ("hopper", "fp16", "fp16"), ("hopper", "e4m3", "fp32"), ("cdna2", "bf16", "fp32")],
                         ids=lambda k: "-".join(k))
def test_one_call_against_three(key):
    from paper_2511_10909_b200 import accuracy, mmasim
    model = mmasim.Model(*key)
    for M, N, K in ((1, 1, 32), (130, 301, 96)):
        A, B, C = (gu.dev(wl.normal_inputs(key[1], key[2], M, N, K, seed=8)[k]) for k in ("A", "B", "C"))
        for c in (C, None):
            got = mmasim.deviation_stats(model, A, B, c)
            ref = accuracy.reference_fp64(key[1], key[2], A, B, c)
            want = mmasim.error_stats(key[2], mmasim.gemm(model, A, B, c), ref).cpu().numpy()
            # FP64 sums of M N terms in another order: at most M N ulps of the sum of magnitudes
            scale = np.maximum(np.abs(want), [1, want[2], 0, 0, 1, 1, 0, 0])
            assert np.all(np.abs(np.array(got) - want) <= M * N * 2.0 ** -52 * scale), (key, (M, N, K), got, want)


# both sizes of tile (1024 x 1100 takes the large ones), K off the kernel's chunk of 16, odd K (copies of eight bytes), infinities and NaNs
@pytest.mark.parametrize("key,sizes", [(("cdna3", "fp16", "fp32"), [(1024, 1100, 72), (130, 301, 72), (129, 65, 7)]), (("hopper", "fp16", "fp16"), [(1024, 1100, 80), (130, 301, 7), (1030, 1100, 5)]),
                                       (("volta", "fp16", "fp16"), [(1024, 1100, 68), (33, 47, 20)]), (("cdna1", "fp32", "fp32"), [(1024, 1100, 71), (100, 90, 33)]),
                                       (("cdna2", "bf16", "fp32"), [(1024, 1100, 36), (70, 33, 36)])], ids=lambda x: "-".join(x) if isinstance(x[0], str) else "")
def test_every_form_of_the_comparing_kernel(key, sizes):
    from paper_2511_10909_b200 import accuracy, mmasim
    model = mmasim.Model(*key)
    top = {"fp16": 0x7C00, "bf16": 0x7F80, "fp32": 0x7F800000}[key[1]]
    for M, N, K in sizes:
        inp = wl.normal_inputs(key[1], key[2], M, N, K, seed=18)
        inp["A"][3, K // 2], inp["A"][7, K - 1], inp["B"][5, 0] = top, top | 1, top
        A, B, C = (gu.dev(inp[k]) for k in ("A", "B", "C"))
        for c in (C, None):
            got = np.array(mmasim.deviation_stats(model, A, B, c))
            ref = accuracy.reference_fp64(key[1], key[2], A, B, c)
            D = mmasim.gemm(model, A, B, c)
            delta = D.view(torch.float16 if key[2] == "fp16" else torch.float32).double() - ref
            counted = int(delta.isfinite().sum())
            assert got[0] == counted <= M * N - 2 * N - M + 2, (key, (M, N, K))
            want = mmasim.error_stats(key[2], D, ref).cpu().numpy()
            # FP64 sums of M N terms in another order: at most M N ulps of the sum of magnitudes
            scale = np.maximum(np.abs(want), [1, want[2], 0, 0, 1, 1, 0, 0])
            assert np.all(np.abs(got - want) <= M * N * 2.0 ** -52 * scale), (key, (M, N, K), got, want)
            assert got[6] == float(delta[delta.isfinite()].abs().max())


def test_operands_that_are_parts_of_larger_ones():
    """Single rows of wider matrices (contiguous whatever their row stride), and a C of more rows and columns than the product has."""
    from paper_2511_10909_b200 import accuracy, mmasim
    key = ("cdna3", "fp16", "fp32")
    model = mmasim.Model(*key)
    inp = wl.normal_inputs(key[1], key[2], 40, 48, 64, seed=9)
    A, B, C = (gu.dev(inp[k]) for k in ("A", "B", "C"))
    wide = torch.nn.functional.pad(A, (0, 32))
    assert accuracy.deviation_stats(model, wide[:1, :64], B, C[:1]) == pytest.approx(accuracy.deviation_stats(model, A[:1].clone(), B, C[:1].clone()), rel=1e-9)
    large = torch.nn.functional.pad(C, (0, 16, 0, 3))
    assert accuracy.deviation_stats(model, A, B, large) == pytest.approx(accuracy.deviation_stats(model, A, B, C), rel=1e-9)


def test_separate_calls_where_the_library_gets_no_memory(monkeypatch):
    """What torch's allocator keeps for itself serves the separate calls; other errors come through."""
    from paper_2511_10909_b200 import accuracy, mmasim
    key = ("hopper", "e4m3", "fp32")
    model = mmasim.Model(*key)
    inp = wl.normal_inputs(key[1], key[2], 40, 48, 64, seed=10)
    A, B, C = (gu.dev(inp[k]) for k in ("A", "B", "C"))
    want = accuracy.deviation_stats(model, A, B, C)

    def fail(message):
        def call(*args, **kw):
            raise mmasim.MmasimError(5, message)
        monkeypatch.setattr(mmasim, "deviation_stats", call)
    fail("mmasim_deviation_stats: out of memory")
    assert accuracy.deviation_stats(model, A, B, C) == pytest.approx(want, rel=1e-9)
    fail("mmasim_deviation_stats: invalid argument")
    with pytest.raises(mmasim.MmasimError):
        accuracy.deviation_stats(model, A, B, C)
